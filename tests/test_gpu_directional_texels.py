"""The directional estimator's projection of triangles onto cube-map texels:
every texel whose ray meets a triangle must be tested.  Face, chunk and queue
edges (one texel a face; several row chunks a face; triangles over whole
faces; centres outside, inside and next to the surface; one box and more
boxes than SMs) against the oracle's FP64 test of every ray and triangle."""
import numpy as np
import pytest

import oracle as O
from synth import meshes as M
from tests import pins

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


def _boxes(m, k, seed, half):
    rng = np.random.Generator(np.random.PCG64(seed))
    V = m.verts.astype(np.float64)
    lo, hi = V.min(0), V.max(0)
    out = np.zeros((k, 12), np.float32)
    for i in range(k):
        R = pins.random_rotation(rng)
        if i % 3 == 0:      # next to the surface
            out[i, :3] = V[rng.integers(len(V))] + rng.normal(scale=0.01, size=3)
        else:
            out[i, :3] = rng.uniform(lo - 0.2, hi + 0.2)
        out[i, 3:6], out[i, 6:9] = R[0], R[1]
        out[i, 9:12] = rng.uniform(*half, 3)
    return out


@pytest.mark.parametrize("shape,m,k", [("cube", 1, 7), ("octahedron", 5, 7), ("cube", 78, 3), ("octahedron", 79, 3),
                                       ("icosphere", 256, 1), ("torus", 31, 6), ("octahedron", 6, 400)])
def test_every_texel_a_triangle_meets_is_tested(ctx, shape, m, k):
    mesh = {"cube": lambda: M.cube(), "octahedron": lambda: M.octahedron(), "icosphere": lambda: M.icosphere(1),
            "torus": lambda: M.torus(1.0, 0.4, 12, 9, jitter=0.01, seed=5)}[shape]()
    boxes = _boxes(mesh, k, 17 + m, (0.1, 0.9))
    h = ctx.mesh_create(mesh.verts, mesh.tris)
    got = ctx.directional_outer_volume(h, boxes, m=m)
    h.free()
    ref = np.array([O.directional_outer_volume(mesh.verts, mesh.tris, b, m=m) for b in boxes])
    # Rounding: a ray's crossings and exit carry below 1e-6 of r_e^3 <= |half|^3, over 4 pi / 3 of solid angle
    # (5e-6 |half|^3); the FP32 solid angles 2.5e-7 a texel, 6 m^2 of them with random signs (below 1e-4 at m = 256).
    # A ray grazing an edge may flip one texel: its cone, at most 4 / m^2 / 3 of |half|^3.
    size = np.linalg.norm(boxes[:, 9:12].astype(np.float64), axis=1) ** 3
    assert np.all(np.abs(got - ref) <= (1e-4 + (1.4 / m ** 2 if m >= 31 else 0.0)) * size)
