"""Covariance frames solved by eight lanes a cluster (few clusters) and by a
thread a cluster (many): the same bits for the same cluster, including flat,
symmetric and degenerate ones; normals of given frames as of solved ones."""
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


@pytest.mark.parametrize("kind,jitter", [("random", 0.004), ("strips", 0.0), ("strips", 0.004), ("flat", 0.0), ("points", 0.0)])
@pytest.mark.parametrize("shared", [1, 3, 4, 997])
def test_frames_do_not_depend_on_the_number_of_clusters(ctx, kind, jitter, shared):
    m = M.torus(1.0, 0.3, 200, 100, jitter=jitter, seed=5)   # 40,000 triangles
    V = np.array(m.verts)
    if kind == "flat":
        V[:, 2] = np.where(V[:, 2] > 0.29, V[:, 2], np.float32(0.25))
    if kind == "points":   # some triangles collapsed to points
        i = m.tris[:300].reshape(-1)
        V[i] = V[i[0]]
    mesh = ctx.mesh_create(V, m.tris)
    lat = ctx.build_occupancy(mesh, 64)
    T = len(m.tris)
    few = np.minimum(np.arange(T) * 2000 // T, 2000 - 1)
    if kind == "random":
        few = np.random.default_rng(1).permutation(few)
    many = few.copy()                                        # the first `shared` clusters stay, the others are cut up
    rest = few >= shared
    many[rest] = shared + np.arange(rest.sum()) % (20000 - shared)
    out = []
    for a in (few, many):
        K = int(a.max()) + 1
        layer = ctx.layer_init(lat, a.astype(np.int32), np.zeros(K, np.int32))
        r = ctx.layer_read(layer)
        layer.free()
        out.append(r)
        # given the same frames, the same boxes
        layer = ctx.layer_init(lat, a.astype(np.int32), np.zeros(K, np.int32), r["frames"])
        assert np.array_equal(ctx.layer_read(layer)["qboxes"], r["qboxes"])
        layer.free()
    assert len(out[0]["frames"]) == 2000 and len(out[1]["frames"]) == 20000
    for key in ("frames", "qboxes", "obv"):
        assert np.array_equal(out[0][key][:shared], out[1][key][:shared]), key
    lat.free()
    mesh.free()


@pytest.mark.parametrize("members", [1, 2, 127, 128, 129, 257, 513, 641, 5000])
def test_frames_do_not_depend_on_how_members_are_loaded(ctx, members):
    """Layers of large clusters load their members ahead; the sums keep their order."""
    m = M.torus(1.0, 0.3, 200, 100, jitter=0.004, seed=8)    # 40,000 triangles
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 64)
    T = len(m.tris)
    pick = np.random.default_rng(members).permutation(T)
    out = []
    for K in (3, 300):                                       # 13,333 and 133 triangles a cluster
        a = np.empty(T, np.int32)
        a[pick[:members]] = 0
        a[pick[members:]] = 1 + np.arange(T - members) % (K - 1)
        layer = ctx.layer_init(lat, a, np.zeros(K, np.int32))
        r = ctx.layer_read(layer)
        out.append([r[key][0] for key in ("frames", "qboxes", "obv")])
        layer.free()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
    lat.free()
    mesh.free()
