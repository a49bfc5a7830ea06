"""Float boxes to integer boxes: entries near and at half-integers, outside the
fast path's range, tiny and zero, boxes that are refused; and the counts of
float boxes against those of the same boxes quantised first."""
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


@pytest.fixture(scope="module", params=["cube", "torus"])
def lat(ctx, request):
    m = M.cube() if request.param == "cube" else M.torus(1.0, 0.3, 60, 24, jitter=0.004, seed=3)
    mesh = ctx.mesh_create(m.verts, m.tris)
    L = ctx.build_occupancy(mesh, 90)
    yield L, np.asarray(m.verts, np.float32)
    L.free()
    mesh.free()


def reference(verts, N, boxes):
    """The definition, a correctly rounded FP64 operation at a time."""
    lo, hi = verts.min(0).astype(np.float64), verts.max(0).astype(np.float64)
    h = (hi - lo) / N
    hm = h.max()
    B = boxes.astype(np.float64)
    c, u, v, half = B[:, :3], B[:, 3:6], B[:, 6:9], B[:, 9:]
    w = np.stack([u[:, 1] * v[:, 2] - u[:, 2] * v[:, 1], u[:, 2] * v[:, 0] - u[:, 0] * v[:, 2],
                  u[:, 0] * v[:, 1] - u[:, 1] * v[:, 0]], 1)
    R = np.stack([u, v, w], 1)
    n = np.rint(R * h / hm * 16777216.0)
    d = c - lo - 0.5 * h
    m = R[:, :, 0] * d[:, None, 0] + R[:, :, 1] * d[:, None, 1] + R[:, :, 2] * d[:, None, 2]
    s = 4294967296.0 / hm
    return n.astype(np.int64), np.stack([np.floor((m - half) * s), np.ceil((m + half) * s)], 2).astype(np.int64)


def boxes_of(rng, K, verts):
    lo, hi = verts.min(0), verts.max(0)
    b = np.zeros((K, 12), np.float32)
    b[:, :3] = rng.uniform(lo, hi, (K, 3))
    R, _ = np.linalg.qr(rng.standard_normal((K, 3, 3)))
    b[:, 3:6], b[:, 6:9] = R[:, 0], R[:, 1]
    b[:, 9:] = rng.uniform(0.0, 0.4, (K, 3)) * (hi - lo)
    return b


def test_entries(ctx, lat):
    L, verts = lat
    rng = np.random.default_rng(5)
    b = boxes_of(rng, 4000, verts)
    half = ((rng.integers(-(1 << 23), 1 << 23, (1000, 3)) + 0.5) / (1 << 24)).astype(np.float32)   # halves, exactly
    b[:1000, 3:6] = half
    b[1000:1400, 3:6] = np.nextafter(half[:400], np.float32(1))
    b[1400:1800, 6:9] = np.nextafter(half[400:800], np.float32(-1))
    b[1800:2000, 3:9] *= 5.0                                                 # |r| >= 2
    b[2000:2200, 3:9] *= rng.choice([1e-6, 1e-9, 1e-30, 1e-44, 0.0, -0.0, 1.9999999], (200, 6)).astype(np.float32)
    b[2200:2300, 3:9] = rng.choice([0.0, -0.0, 1.0, -1.0, 2.0, -2.0, 1.5], (100, 6))
    b[2300:2350, 9:] = 0.0
    q = ctx.quantize_boxes(L, b)
    n, bounds = reference(verts, 90, b)
    assert np.abs(n).max() < 2 ** 31
    assert np.array_equal(q["n"].reshape(-1, 9), n.reshape(-1, 9))
    assert np.array_equal(q["b"].reshape(-1, 6), bounds.reshape(-1, 6))


def test_refused_boxes(ctx, lat):
    L, verts = lat
    for K in (1, 40):
        for col, val in ((0, np.nan), (4, np.inf), (11, -1e-3), (9, np.nan), (1, 1e30)):
            b = boxes_of(np.random.default_rng(col), K, verts)
            b[K - 1, col] = val
            with pytest.raises(Exception):
                ctx.quantize_boxes(L, b)
            with pytest.raises(Exception):
                ctx.outer_volume(L, b)


@pytest.mark.parametrize("K", [1, 31, 33, 512, 513, 1025, 4096, 4097])
def test_float_boxes_count_as_quantised_ones(ctx, lat, K):
    L, verts = lat
    b = boxes_of(np.random.default_rng(K), K, verts)
    a = ctx.outer_volume(L, b, want_points=True)
    c = ctx.outer_volume_q(L, ctx.quantize_boxes(L, b), want_points=True)
    for x, y in zip(a, c):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("K", [2, 9, 33, 600])
@pytest.mark.parametrize("every", [1, 2, 3, 8])
def test_empty_boxes_among_others(ctx, lat, K, every):
    """Boxes without a point, axis-aligned ones and rotated ones prepared by one warp."""
    L, verts = lat
    b = boxes_of(np.random.default_rng(K + every), K, verts)
    b[::every, 9:] = 0.0                                       # no lattice point inside, unless by chance
    b[1::5, 3:9] = np.r_[1.0, 0, 0, 0, 1, 0]
    q = ctx.quantize_boxes(L, b)
    got = ctx.outer_volume(L, b, want_points=True)
    again = ctx.outer_volume_q(L, q, want_points=True)
    one = [ctx.outer_volume_q(L, q[k:k + 1], want_points=True) for k in range(min(K, 40))]
    for i in range(2):
        assert np.array_equal(got[i], again[i])
        assert np.array_equal(got[i][:len(one)], np.concatenate([o[i] for o in one]))
    assert np.all(got[0][::every] <= 8)
