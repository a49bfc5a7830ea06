"""A box's features do not depend on the batch it comes in: batches of blocks of
eight boxes and of thirty-two, whole and partial blocks, a lattice edge."""
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


@pytest.mark.parametrize("k", [1, 7, 8, 9, 32, 33, 255, 4863])
def test_features_of_a_batch_are_those_of_a_larger_one(ctx, k):
    m = M.sdf_union_mesh(7, 14, n_spheres=6, n_capsules=3)
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 67)
    q = np.resize(ctx.quantize_boxes(lat, _boxes(m, 257, 5)), 20000)     # beyond the line on any chip
    assert np.array_equal(ctx.surrogate_features(lat, q[:k]), ctx.surrogate_features(lat, q)[:k])
    lat.free()
    mesh.free()
