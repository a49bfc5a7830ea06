"""Median splits: clusters whose median a block selects and clusters that are
sorted, with many equal keys (ties by triangle), against an ordering of all
triangles by (cluster, key, triangle)."""
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


def folded(nx, ny):
    """A closed strip that runs out along x and back: 4 ny triangles share each pair of x coordinates."""
    i, j = np.meshgrid(np.arange(nx), np.arange(ny), indexing="ij")
    a = 2 * np.pi * j / ny
    v = np.stack([np.minimum(i, nx - i) / nx, 0.2 * np.cos(a), 0.2 * np.sin(a) + 0.01 * (i > nx // 2)], -1)
    i, j = i.ravel(), j.ravel()
    at = lambda p, q: (p % nx) * ny + q % ny
    a, b, c, d = at(i, j), at(i + 1, j), at(i, j + 1), at(i + 1, j + 1)
    f = np.concatenate([np.stack([a, b, c], 1), np.stack([b, d, c], 1)])
    return v.reshape(-1, 3).astype(np.float32), f.astype(np.int32)


def expected(lat, tris, assign, q):
    U = lat.fixed().cpu().numpy().astype(np.int64)
    s = U[tris].sum(1)
    n = q["n"].reshape(-1, 9)[:, :3].astype(np.int64)
    key = (n[assign] * s).sum(1)
    order = np.lexsort((np.arange(len(tris)), key, assign))
    size = np.bincount(assign)
    start = np.concatenate([[0], np.cumsum(size)])
    rank = np.empty(len(tris), np.int64)
    rank[order] = np.arange(len(tris)) - start[assign[order]]
    return (2 * assign + (rank >= (size[assign] + 1) // 2)).astype(np.int32)


# (steps along x, around it, clusters): columns of up to 4,000 equal keys, blocks of 256 and of 1,024 threads, clusters
# of 2 to 256 and of more triangles, clusters that are sorted (more than 131,072 triangles)
@pytest.mark.parametrize("nx,ny,K", [(10, 600, 1), (4, 1000, 1), (40, 600, 24), (64, 3, 192), (64, 128, 64), (64, 128, 1),
                                     (64, 129, 1), (8, 16, 1), (3, 43, 1), (129, 3, 3), (300, 300, 1), (300, 300, 11),
                                     (300, 300, 400), (256, 256, 1)])
def test_split_is_the_median(ctx, nx, ny, K):
    v, f = folded(nx, ny)
    mesh = ctx.mesh_create(v, f)
    lat = ctx.build_occupancy(mesh, 64)
    T = len(f)
    rng = np.random.default_rng(nx + ny + K)
    for assign in (np.arange(T) * K // T, rng.permutation(np.arange(T) % K)):
        assign = assign.astype(np.int32)
        frames = np.tile(np.eye(3), (K, 1, 1))
        frames[1::3] = -frames[1::3]
        layer = ctx.layer_init(lat, assign, np.zeros(K, np.int32), frames)
        q = ctx.layer_read(layer)["qboxes"]
        assert np.array_equal(ctx.layer_split(layer), expected(lat, f, assign, q))
        layer.free()
    lat.free()
    mesh.free()


@pytest.mark.parametrize("level,rounds", [(1, 1), (3, 2), (9, 1)])
def test_split_after_rounds_that_ended_moving(ctx, level, rounds):
    m = M.torus(1.0, 0.3, 60, 24, jitter=0.004, seed=7)
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 64)
    tree = ctx.build_tree(lat, level, 0)
    r = ctx.tree_read(tree, level)
    for parent in (np.arange(1 << level) // 2, np.zeros(1 << level)):
        layer = ctx.layer_init(lat, r["assign"], parent.astype(np.int32), r["frames"])
        ctx.lloyd_step(layer, rounds=rounds, refit=0)
        now = ctx.layer_read(layer)
        try:
            got = ctx.layer_split(layer)
        except Exception as e:   # a cluster left with one triangle is refused
            assert np.bincount(now["assign"]).min() < 2, e
        else:
            assert np.array_equal(got, expected(lat, m.tris, now["assign"], now["qboxes"]))
        layer.free()
    for x in (tree, lat, mesh):
        x.free()


def test_split_of_one_triangle_is_refused(ctx):
    v, f = folded(8, 8)
    mesh = ctx.mesh_create(v, f)
    lat = ctx.build_occupancy(mesh, 32)
    assign = np.r_[0, np.ones(len(f) - 1)].astype(np.int32)
    layer = ctx.layer_init(lat, assign, np.zeros(2, np.int32))
    with pytest.raises(Exception):
        ctx.layer_split(layer)
    layer.free()
    lat.free()
    mesh.free()
