"""Boxes near the longest that a count accepts: a tile of 32 lanes and up to
128 rows a lane of more than a million points each holds more than 2^32
points."""
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
def lat(ctx):
    m = M.torus(1.0, 0.3, 24, 12)
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 16)
    yield lat
    lat.free()
    mesh.free()


def _boxes(K, n, lo, hi):
    """K one-point boxes, the last replaced by the box of the integer normals n and index bounds lo, hi (times n's 2^24)."""
    import paper_2203_10521_gb300 as P
    q = np.zeros(K, P.QBOX_DTYPE)
    q["n"] = (np.eye(3, dtype=np.int64) << 24).reshape(9)
    q["n"][-1] = np.asarray(n).reshape(9)
    q["b"][-1, 0::2] = np.asarray(lo, np.int64) << 32
    q["b"][-1, 1::2] = np.asarray(hi, np.int64) << 32
    return q


# more than 512 boxes take the general path with tiles of full height; lengths around 2^32 points a tile of 128 rows a
# lane and the longest accepted (the bounding box's margin is a few cells of 2^20)
@pytest.mark.parametrize("tile", [32, 64, 128])
@pytest.mark.parametrize("length", [(1 << 20) - 200, (1 << 20) + 77, (1 << 21) - 160])
@pytest.mark.parametrize("axis", [0, 1])
def test_long_rows_of_a_tall_tile(ctx, lat, tile, length, axis):
    import torch
    lo, hi = [-72, -72, -72], [90, 87, 95]                    # 160 x 168 rows or more, around the whole lattice
    lo[axis], hi[axis] = -(length // 2), length - length // 2 - 1
    q = _boxes(600, np.eye(3, dtype=np.int64) << 24, lo, hi)
    points = int(np.prod([b - a + 1 for a, b in zip(lo, hi)], dtype=np.int64))
    empty = points - int(np.unpackbits(np.asarray(lat.words().cpu().numpy()).view(np.uint8)).sum())
    ctx.set_counting_tile(tile)
    ctx.set_counting_axis(axis)
    try:
        counts, pts = ctx.outer_volume_q(lat, q, want_points=True)
        one, one_pts = ctx.outer_volume_q(lat, q[-1:], want_points=True)
        dq = torch.from_numpy(q.view(np.uint8).copy()).cuda()
        nc, npt = (torch.zeros(len(q), dtype=torch.int64, device="cuda") for _ in range(2))
        ctx.outer_volume_q_noalloc(lat, dq, nc, npt)
    finally:
        ctx.set_counting_tile(32)
        ctx.set_counting_axis(0)
    assert (int(one[0]), int(one_pts[0])) == (empty, points)
    assert (int(counts[-1]), int(pts[-1])) == (empty, points)
    assert (int(nc[-1]), int(npt[-1])) == (empty, points)


@pytest.mark.parametrize("tile", [64, 128])
def test_long_rows_of_a_slightly_turned_box(ctx, lat, tile):
    """All three slabs step along the rows (no band, no slab almost parallel to them)."""
    s = 160                                                   # 10^-5 of 2^24: 20 rows over the box's length
    n = np.array([[1 << 24, s, -s], [-s, 1 << 24, s], [s, -s, 1 << 24]])
    q = _boxes(600, n, [-(1 << 20) + 400, -90, -90], [(1 << 20) - 400, 90, 90])
    ctx.set_counting_tile(tile)
    ctx.set_counting_axis(0)
    try:
        counts, pts = ctx.outer_volume_q(lat, q, want_points=True)
        one, one_pts = ctx.outer_volume_q(lat, q[-1:], want_points=True)
    finally:
        ctx.set_counting_tile(32)
        ctx.set_counting_axis(0)
    assert int(one_pts[0]) > 180 * 180 * ((1 << 21) - 1000)
    assert (int(counts[-1]), int(pts[-1])) == (int(one[0]), int(one_pts[0]))
