"""Exact flooding of large boxes by few triangles goes a wave per launch, other
exact flooding by a cluster per group: the same partition, many or few
launches."""
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


# N^3 <= 6 10^7 sqrt(triangles): 36 triangles up to 711^3, 144 up to 896^3
@pytest.mark.parametrize("nu,nv,N,by_groups", [(6, 3, 700, True), (6, 3, 720, False), (12, 6, 880, True),
                                               (12, 6, 910, False)])
def test_large_boxes_flood_in_waves(ctx, nu, nv, N, by_groups):
    m = M.torus(1.0, 0.3, nu, nv, jitter=0.004, seed=9)
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, N)
    tree = ctx.build_tree(lat, 3, 0)
    r = ctx.tree_read(tree, 3)
    parent = (np.arange(8) // 2).astype(np.int32)
    out = []
    for mode in (0, 1):          # profiling with counters always goes a wave per launch
        layer = ctx.layer_init(lat, r["assign"], parent, r["frames"])
        ctx.profile_enable(mode)
        n0 = ctx.profile_read()["launches"]
        st = ctx.flood_partition(layer, mode=0)
        out.append((st, ctx.profile_read()["launches"] - n0, ctx.layer_read(layer)))
        ctx.profile_enable(0)
        layer.free()
    (sa, na, a), (sb, nb, b) = out
    assert sa == sb
    for k in ("assign", "qboxes", "obv"):
        assert np.array_equal(a[k], b[k]), k
    waves = sa["waves"]
    assert waves >= 4 and (na + 3 * waves < nb if by_groups else na == nb)
    for x in (tree, lat, mesh):
        x.free()
