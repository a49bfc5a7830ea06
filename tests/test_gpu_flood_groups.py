"""Exact flooding by a cluster per group against the same flooding a wave per
launch (which profiled calls take): group sizes from one box to eight, uneven
groups, a group longer than one launch takes, many small groups."""
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
def torus(ctx):
    m = M.torus(1.0, 0.3, 90, 30, jitter=0.002, seed=3)     # 5,400 triangles
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 61)
    tree = ctx.build_tree(lat, 7, 0)
    levels = [ctx.tree_read(tree, lev) for lev in range(8)]
    tree.free()
    yield lat, levels
    lat.free()
    mesh.free()


@pytest.mark.parametrize("level,parent", [(0, lambda k: k), (1, lambda k: k // 2), (3, lambda k: k // 8),
                                          (3, lambda k: np.where(k < 5, 6, 2)), (5, lambda k: (k * 7) % 9),
                                          (7, lambda k: k // 2)])
def test_groups_equal_waves(ctx, torus, level, parent):
    lat, levels = torus
    L = levels[level]
    p = parent(np.arange(1 << level)).astype(np.int32)
    out = []
    for prof in (0, 2):
        layer = ctx.layer_init(lat, L["assign"], p, L["frames"])
        ctx.profile_enable(prof)
        try:
            st = ctx.flood_partition(layer, mode=0)
        finally:
            ctx.profile_enable(0)
        out.append((st, ctx.layer_read(layer)))
        layer.free()
    (sa, a), (sb, b) = out
    assert sa == sb
    assert np.array_equal(a["assign"], b["assign"]) and np.array_equal(a["obv"], b["obv"])
    assert np.array_equal(a["qboxes"], b["qboxes"])
