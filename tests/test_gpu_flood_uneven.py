"""Exact flooding of many uneven groups: the cluster of the long ones grows as
the short ones end (several launches), the partition is that of the waves."""
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


# 125 groups of four (the longest has 4,800 of 24,000 triangles), 300 of two, 38 (eight blocks each from the start),
# groups of like size (one launch)
@pytest.mark.parametrize("K,per,power,grows", [(500, 4, 3, True), (600, 2, 3, True), (76, 2, 3, False), (500, 4, 1, False)])
def test_uneven_groups_equal_waves(ctx, K, per, power, grows):
    m = M.torus(1.0, 0.3, 200, 60, jitter=0.004, seed=3)
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 64)
    T = len(m.tris)
    parent = (np.arange(K) // per).astype(np.int32)

    def flood(power, mode):
        a = np.minimum(np.floor(K * (np.arange(T) / T) ** power).astype(int), K - 1)
        a[:K] = np.arange(K)
        layer = ctx.layer_init(lat, a.astype(np.int32), parent)
        ctx.profile_enable(mode)
        n0 = ctx.profile_read()["launches"]
        st = ctx.flood_partition(layer, mode=0)
        n = ctx.profile_read()["launches"] - n0
        r = ctx.layer_read(layer)
        ctx.profile_enable(0)
        layer.free()
        return st, n - -(-st["waves"] // 4096), r      # without the orders' launches

    (sa, na, x), (sb, _, y) = flood(power, 0), flood(power, 1)   # profiling with counters goes a wave per launch
    assert sa == sb
    for k in ("assign", "qboxes", "obv"):
        assert np.array_equal(x[k], y[k]), k
    extra = na - flood(1, 0)[1]       # against groups of like size: lists of the unfinished and further runs
    assert extra >= 2 if grows else extra == 2 * (sa["waves"] // 4096)
    lat.free()
    mesh.free()
