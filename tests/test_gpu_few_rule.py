"""Up to 96 boxes on a small lattice are counted in one launch, more in two: the
same counts on both sides of the line, in every form of a call."""
import numpy as np
import pytest

from synth import meshes as M
from tests.test_gpu_few_boxes import _boxes

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


@pytest.mark.parametrize("N", [17, 64])
@pytest.mark.parametrize("k,launches", [(1, 1), (96, 1), (97, 2), (400, 2)])
def test_launches_of_a_count(ctx, N, k, launches):
    m = M.sdf_union_mesh(7, 14, n_spheres=6, n_capsules=3)
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, N)
    boxes = _boxes(m, k, 100 + k)
    q = ctx.quantize_boxes(lat, boxes)
    ctx.profile_enable(1)                  # the general path with its counters
    want = ctx.outer_volume_q(lat, q, want_points=True)
    ctx.profile_enable(0)
    for call in (lambda: ctx.outer_volume(lat, boxes, want_points=True), lambda: ctx.outer_volume_q(lat, q, want_points=True)):
        n0 = ctx.profile_read()["launches"]
        got = call()
        assert ctx.profile_read()["launches"] - n0 == launches
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    lat.free()
    mesh.free()
