"""Few boxes on a small lattice are counted in one launch, a cluster per box;
other calls of few boxes with shorter tiles and offsets scanned by the
preparation's last block; profiled ones by the general path with full tiles.
All give the same counts, points and errors for every form of a call."""
import numpy as np
import pytest

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


@pytest.fixture(scope="module")
def lats(ctx):
    m = M.sdf_union_mesh(7, 14, n_spheres=6, n_capsules=3)
    mesh = ctx.mesh_create(m.verts, m.tris)
    ctx.set_counting_axis(-1)      # keep the y- and z-row copies
    out = [ctx.build_occupancy(mesh, n) for n in (67, 200)]
    ctx.set_counting_axis(0)
    yield m, out
    for x in out:
        x.free()
    mesh.free()


def _boxes(m, k, seed):
    """Rotated, axis-aligned and flat boxes from a cell to beyond the lattice."""
    rng = np.random.Generator(np.random.PCG64(seed))
    lo, hi = m.verts.min(0).astype(np.float64), m.verts.max(0).astype(np.float64)
    out = np.zeros((k, 12), np.float32)
    for i in range(k):
        R = np.eye(3) if i % 5 == 0 else pins.random_rotation(rng)
        out[i, :3] = rng.uniform(lo - 0.2, hi + 0.2)
        out[i, 3:6], out[i, 6:9] = R[0], R[1]
        out[i, 9:12] = np.exp(rng.uniform(np.log(0.005), np.log(1.5), 3))
        if i % 7 == 3:
            out[i, 9] = 0.0
    return out


def _general(ctx, f):
    ctx.profile_enable(2)          # events only: the general path
    try:
        return f()
    finally:
        ctx.profile_enable(0)


@pytest.mark.parametrize("k", [1, 2, 63, 512])
@pytest.mark.parametrize("tile,axis,rank", [(32, 0, 1), (1, -1, 1), (128, 2, 0)])
def test_one_launch_counts_equal_the_general_path(ctx, lats, k, tile, axis, rank):
    import torch
    m, (small, large) = lats
    boxes = _boxes(m, k, 100 + k)
    ctx.set_counting_tile(tile)
    ctx.set_counting_axis(axis)
    ctx.set_counting_rank(rank)
    try:
        for lat in (small, large):
            q = ctx.quantize_boxes(lat, boxes)
            dq = torch.from_numpy(q.view(np.uint8).copy()).cuda()
            ref = _general(ctx, lambda: ctx.outer_volume_q(lat, q, want_points=True))
            for got in (ctx.outer_volume(lat, boxes, want_points=True), ctx.outer_volume_q(lat, q, want_points=True),
                        [x.cpu().numpy().view(np.uint64) for x in ctx.outer_volume_q(lat, dq, want_points=True)]):
                assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
            assert np.array_equal(ctx.outer_volume(lat, boxes), ref[0])
        which = (np.arange(k) % 2).astype(np.int32)
        q2 = np.concatenate([ctx.quantize_boxes(lats[1][w], boxes[i:i + 1]) for i, w in enumerate(which)])
        a = ctx.outer_volume_multi([small, large], q2, which, want_points=True)
        b = _general(ctx, lambda: ctx.outer_volume_multi([small, large], q2, which, want_points=True))
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    finally:
        ctx.set_counting_tile(32)
        ctx.set_counting_axis(0)
        ctx.set_counting_rank(1)


@pytest.mark.parametrize("field,value", [(0, np.nan), (10, -0.1), (4, np.inf), (9, 1e30)])
def test_one_launch_reports_bad_boxes(ctx, lats, field, value):
    m, (small, _) = lats
    import paper_2203_10521_gb300 as P
    boxes = _boxes(m, 6, 9)
    good = ctx.outer_volume(small, boxes)
    bad = boxes.copy()
    bad[2, field] = value
    codes = []
    for f in (lambda: ctx.outer_volume(small, bad), lambda: _general(ctx, lambda: ctx.outer_volume(small, bad))):
        with pytest.raises(P.ObbError) as e:
            f()
        codes.append(e.value.code)
    assert codes[0] == codes[1]
    assert np.array_equal(ctx.outer_volume(small, boxes), good)     # the context stays usable
