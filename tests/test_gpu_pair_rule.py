"""Which layers of sibling pairs run their rounds pair by pair (few launches a
step) and which as the layer's rounds, and that the results do not tell."""
import numpy as np
import pytest

from synth import meshes as M

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2203_10521_gb300 as P
    c = P.Context(0)
    yield c
    torch.cuda.synchronize()
    c.close()


def _step(ctx, layer, **kw):
    n0 = ctx.profile_read()["launches"]
    st = ctx.lloyd_step(layer, **kw)
    return st, ctx.profile_read()["launches"] - n0


# N^2 <= 65,536 pairs + 32 triangles: both sides of the line by lattice, by pairs and by triangles
@pytest.mark.parametrize("nu,nv,N,level,by_pairs", [(60, 16, 350, 1, True), (60, 16, 360, 1, False),
                                                    (60, 16, 568, 3, True), (60, 16, 700, 3, False),
                                                    (200, 100, 700, 1, True)])
def test_large_boxes_of_few_pairs_take_the_layer_rounds(ctx, nu, nv, N, level, by_pairs):
    m = M.torus(1.0, 0.3, nu, nv, jitter=0.004, seed=9)
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, N)
    tree = ctx.build_tree(lat, level, 0)
    r = ctx.tree_read(tree, level)
    parent = (np.arange(1 << level) // 2).astype(np.int32)
    out = []
    for mode in (0, 1):          # profiling with counters always takes the layer's
        layer = ctx.layer_init(lat, r["assign"], parent, r["frames"])
        ctx.profile_enable(mode)
        st, n = _step(ctx, layer, rounds=16, refit=0)
        ctx.profile_enable(0)
        out.append((st, n, ctx.layer_read(layer)))
        layer.free()
    (sa, na, a), (sb, nb, b) = out
    assert sa == sb
    for k in ("assign", "qboxes", "obv"):
        assert np.array_equal(a[k], b[k]), k
    assert (na < nb) == by_pairs and (na == nb) != by_pairs
    for x in (tree, lat, mesh):
        x.free()


@pytest.mark.parametrize("graph,N,level,switches", [(False, 513, 8, True), (True, 513, 8, True), (False, 512, 8, False),
                                                    (True, 512, 8, False), (False, 560, 7, True)])
def test_settled_large_layers_take_their_own_rounds(ctx, graph, N, level, switches):
    """Above 512^3, unless of large clusters: after one step without a move, two when captured; a move takes them back."""
    m = M.torus(1.0, 0.3, 90, 30, jitter=0.004, seed=3)      # 5,400 triangles
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, N)
    tree = ctx.build_tree(lat, level, 0)
    r = ctx.tree_read(tree, level)
    parent = (np.arange(1 << level) // 2).astype(np.int32)
    a = ctx.layer_init(lat, r["assign"], parent, r["frames"])
    b = ctx.layer_init(lat, r["assign"], parent, r["frames"])
    launches, quiet = [], 0
    for _ in range(40):
        st, n = _step(ctx, a, rounds=16, refit=0, graph=graph)
        ctx.profile_enable(1)
        assert st == ctx.lloyd_step(b, rounds=16, refit=0)   # by the layer's rounds
        ctx.profile_enable(0)
        quiet = quiet + 1 if st["moves"] == 0 else 0
        launches.append((quiet, n))
        if quiet == 5:
            break
    assert quiet == 5 and launches[0][0] == 0
    by_pairs = launches[0][1]
    assert by_pairs < 6
    for q, n in launches:
        later = q > (2 if graph else 1)
        assert (n > by_pairs) == (switches and later), launches
    # the layer changes: pairs again, and the same results
    for x in (a, b):
        ctx.flood_partition(x, mode=0)
    st, n = _step(ctx, a, rounds=16, refit=0, graph=graph)
    ctx.profile_enable(1)
    assert st == ctx.lloyd_step(b, rounds=16, refit=0) and st["moves"] > 0
    ctx.profile_enable(0)
    st2, n2 = _step(ctx, a, rounds=1, refit=0, graph=graph)
    assert n2 == by_pairs
    ctx.lloyd_step(b, rounds=1, refit=0)
    x, y = ctx.layer_read(a), ctx.layer_read(b)
    for k in ("assign", "qboxes", "obv"):
        assert np.array_equal(x[k], y[k]), k
    for z in (a, b, tree, lat, mesh):
        z.free()


@pytest.mark.parametrize("kind,by_pairs", [("split", True), ("scattered", False), ("swapped", False)])
@pytest.mark.parametrize("graph", [False, True])
def test_a_huge_box_takes_the_layer_to_its_own_rounds(ctx, kind, by_pairs, graph):
    """The same lattice and number of pairs: compact clusters, scattered ones, and two triangles of distant clusters
    exchanged (two boxes across the whole model)."""
    m = M.torus(1.0, 0.3, 200, 60, jitter=0.004, seed=3)     # 24,000 triangles
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 1000)
    tree = ctx.build_tree(lat, 9, 0)
    a = ctx.tree_read(tree, 9)["assign"].copy()
    if kind == "scattered":
        a = np.random.default_rng(1).permutation(a)
    elif kind == "swapped":
        c = np.asarray(m.verts)[m.tris].mean(1)
        i = int(c.sum(1).argmin())
        j = int(c.sum(1).argmax())           # opposite ends of the model
        a[i], a[j] = a[j], a[i]
    parent = (np.arange(512) // 2).astype(np.int32)
    out = []
    for mode in (0, 1):
        layer = ctx.layer_init(lat, a, parent)
        ctx.profile_enable(mode)
        # (a captured step in mode 1 would be the same graph)
        steps = [_step(ctx, layer, rounds=16, refit=1, graph=graph and mode == 0) for _ in range(2)]
        ctx.profile_enable(0)
        out.append((steps, ctx.layer_read(layer)))
        layer.free()
    (sa, x), (sb, y) = out
    assert [s for s, _ in sa] == [s for s, _ in sb]
    for k in ("assign", "qboxes", "obv", "frames"):
        assert np.array_equal(x[k], y[k]), k
    rounds = sa[0][0]["rounds_run"]
    assert (sa[0][1] < 7 + 7 * rounds) == by_pairs           # a round by the layer is at least seven launches
    for z in (tree, lat, mesh):
        z.free()
