"""A layer's moments are those that its refit sums: layers of large clusters
through the kernel that loads members ahead, with the same bits as without
(the precision test compares both with FP64)."""
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


@pytest.mark.parametrize("members", [1, 127, 129, 385, 513, 641, 6007])
def test_moments_of_one_cluster_in_large_and_small_company(ctx, members):
    m = M.torus(1.0, 0.3, 200, 100, jitter=0.004, seed=8)    # 40,000 triangles
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 64)
    T = len(m.tris)
    pick = np.random.default_rng(members).permutation(T)
    got = []
    for K in (3, 300):                                       # 13,333 and 133 triangles a cluster: ahead, and not
        a = np.empty(T, np.int32)
        a[pick[:members]] = 0
        a[pick[members:]] = 1 + np.arange(T - members) % (K - 1)
        layer = ctx.layer_init(lat, a, np.zeros(K, np.int32))
        got.append(ctx.layer_moments(layer, compensated=True)[0])
        layer.free()
    assert np.array_equal(got[0], got[1])
    lat.free()
    mesh.free()
