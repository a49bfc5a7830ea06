"""Partition rounds pair by pair against the rounds of the whole layer (which
profiled calls take): pairs from one to more than the chip holds at once, one-
triangle clusters, round limits that cut moves short, and what the step
leaves behind (members, candidates, counters)."""
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


@pytest.fixture(scope="module")
def torus(ctx):
    m = M.torus(1.0, 0.3, 120, 36, jitter=0.004, seed=9)     # 8,640 triangles
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 75)
    tree = ctx.build_tree(lat, 12, 0)
    levels = [ctx.tree_read(tree, lev) for lev in range(13)]
    tree.free()
    yield lat, levels
    lat.free()
    mesh.free()


def _same(a, b):
    for k in a:
        assert np.array_equal(a[k], b[k]), k


def _step(ctx, layer, prof, **kw):
    ctx.profile_enable(prof)
    try:
        return ctx.lloyd_step(layer, **kw)
    finally:
        ctx.profile_enable(0)


def _sorted(q, c):
    r = np.concatenate([q.view(np.uint8).reshape(len(q), -1), c.view(np.uint8).reshape(len(c), -1)], 1)
    return r[np.lexsort(r.T)]


# 1 to 2,048 pairs: 8 blocks of 128 threads, 256 threads, one block of 128; level 12: clusters of two triangles
@pytest.mark.parametrize("level,rounds,refit", [(1, 16, 1), (2, 1, 0), (5, 3, 1), (7, 16, 3), (8, 64, 0), (9, 2, 1),
                                                (11, 16, 1), (12, 16, 2), (3, 65, 0)])
def test_pairs_equal_rounds(ctx, torus, level, rounds, refit):
    lat, levels = torus
    L = levels[level]
    parent = (np.arange(1 << level) // 2).astype(np.int32)
    a = ctx.layer_init(lat, L["assign"], parent, L["frames"])
    b = ctx.layer_init(lat, L["assign"], parent, L["frames"])
    g = ctx.layer_init(lat, L["assign"], parent, L["frames"])
    moves = 0
    for it in range(3):
        sa = _step(ctx, a, 0, rounds=rounds, refit=refit)
        sb = _step(ctx, b, 2, rounds=rounds, refit=refit)
        sg = _step(ctx, g, 0, rounds=rounds, refit=refit, graph=True)
        assert sa == sb == sg
        moves += sa["moves"]
        _same(ctx.layer_read(a), ctx.layer_read(b))
        _same(ctx.layer_read(a), ctx.layer_read(g))
        for x, y in zip(ctx.layer_members(a), ctx.layer_members(b)):
            assert np.array_equal(x, y)
        assert np.array_equal(_sorted(*ctx.layer_last_candidates(a)), _sorted(*ctx.layer_last_candidates(b)))
    assert moves > 0
    # a layer may change its way between steps
    sa = _step(ctx, a, 2, rounds=rounds, refit=1)
    sb = _step(ctx, b, 0, rounds=rounds, refit=1)
    assert sa == sb
    _same(ctx.layer_read(a), ctx.layer_read(b))
    for x in (a, b, g):
        x.free()


@pytest.mark.parametrize("parent", [lambda k: k // 4, lambda k: 99 - k // 2, lambda k: (k + 1) // 2, lambda k: 0 * k])
def test_other_sibling_structures_take_the_layer_rounds(ctx, torus, parent):
    """Parents that are not ascending pairs: the same call, by the layer's rounds."""
    lat, levels = torus
    L = levels[4]
    p = parent(np.arange(16)).astype(np.int32)
    out = []
    for prof in (0, 2):
        layer = ctx.layer_init(lat, L["assign"], p, L["frames"])
        out.append((_step(ctx, layer, prof, rounds=8, refit=1), ctx.layer_read(layer)))
        layer.free()
    assert out[0][0] == out[1][0]
    _same(out[0][1], out[1][1])


@pytest.mark.parametrize("upper", [1, 2, 3, 4, 6, 8])
def test_parents_changed_by_a_unit_step(ctx, torus, upper):
    """A unit step may move boxes between parents: the lower layer's next step must see the new ones."""
    lat, levels = torus
    out = []
    for prof in (0, 2):
        K = 1 << upper
        up = ctx.layer_init(lat, levels[upper]["assign"], (np.arange(K) // 2).astype(np.int32), levels[upper]["frames"])
        low = ctx.layer_init(lat, levels[upper + 1]["assign"], (np.arange(2 * K) // 2).astype(np.int32),
                             levels[upper + 1]["frames"])
        st = [_step(ctx, low, prof, rounds=1, refit=0)]
        ctx.profile_enable(prof)
        st.append(ctx.unit_step(up, low, rounds=4))
        ctx.profile_enable(0)
        st.append(_step(ctx, low, prof, rounds=8, refit=1))
        out.append((st, ctx.layer_parents(low), ctx.layer_read(low)))
        up.free()
        low.free()
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1])
    _same(out[0][2], out[1][2])


@pytest.mark.parametrize("level", [1, 2, 3])
def test_few_pairs_on_a_large_lattice(ctx, level):
    """Two pairs or fewer at 257^3 take wider blocks, four do not."""
    m = M.torus(1.0, 0.3, 60, 24, jitter=0.004, seed=11)
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 257)
    tree = ctx.build_tree(lat, level, 0)
    r = ctx.tree_read(tree, level)
    parent = (np.arange(1 << level) // 2).astype(np.int32)
    out = []
    for prof in (0, 2):
        layer = ctx.layer_init(lat, r["assign"], parent, r["frames"])
        out.append((_step(ctx, layer, prof, rounds=6, refit=2), ctx.layer_read(layer)))
        layer.free()
    assert out[0][0] == out[1][0]
    _same(out[0][1], out[1][1])
    for x in (tree, lat, mesh):
        x.free()


@pytest.mark.parametrize("depth", [0, 1, 9, 13])
def test_tree_score_is_the_weighted_sum_of_its_levels(ctx, torus, depth):
    lat, _ = torus
    tree = ctx.build_tree(lat, depth, 0)
    want = sum((depth - lev + 1) * int(ctx.tree_read(tree, lev)["obv"].sum()) for lev in range(depth + 1))
    assert ctx.tree_score(tree)[0] == want
    tree.free()


@pytest.mark.parametrize("level,refit", [(1, 1), (2, 3), (3, 2), (4, 1)])
def test_captured_rounds_of_few_large_pairs(ctx, level, refit):
    """20,000 to 5,000 triangles a cluster take the pairs' rounds in a graph too, 2,500 do not."""
    m = M.torus(1.0, 0.3, 200, 100, jitter=0.004, seed=10)
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 90)
    tree = ctx.build_tree(lat, level, 0)
    r = ctx.tree_read(tree, level)
    parent = (np.arange(1 << level) // 2).astype(np.int32)
    layers = [ctx.layer_init(lat, r["assign"], parent, r["frames"]) for _ in range(3)]
    for it in range(3):
        st = [_step(ctx, layers[0], 0, rounds=16, refit=refit), _step(ctx, layers[1], 2, rounds=16, refit=refit),
              _step(ctx, layers[2], 0, rounds=16, refit=refit, graph=True)]
        assert st[0] == st[1] == st[2]
        for x in layers[1:]:
            _same(ctx.layer_read(layers[0]), ctx.layer_read(x))
    for x in layers + [tree, lat, mesh]:
        x.free()
