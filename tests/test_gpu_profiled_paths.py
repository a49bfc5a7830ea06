"""Profiling that only times (mode 2) runs what an unprofiled call runs;
profiling with counters (mode 1) takes the other paths (a counting launch per
count, the layer's rounds, a wave of flooding per launch), which the tests of
the default paths are repeated against."""
import numpy as np
import pytest

from synth import meshes as M
from tests import test_gpu_few_boxes as few
from tests import test_gpu_flood_groups as groups
from tests import test_gpu_pair_rounds as pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2203_10521_gb300 as P

    class Counters(P.Context):
        """Where a test asks for events alone to leave the default path, counters."""
        def profile_enable(self, on=True):
            super().profile_enable(1 if on == 2 else on)

        def profile_times(self):
            super().profile_enable(2)

    c = Counters(0)
    yield c
    torch.cuda.synchronize()
    c.close()


lats = few.lats
torus = pairs.torus
flood_torus = groups.torus
test_one_launch_counts_equal_the_general_path = few.test_one_launch_counts_equal_the_general_path
test_pairs_equal_rounds = pairs.test_pairs_equal_rounds
test_other_sibling_structures_take_the_layer_rounds = pairs.test_other_sibling_structures_take_the_layer_rounds
test_parents_changed_by_a_unit_step = pairs.test_parents_changed_by_a_unit_step
test_few_pairs_on_a_large_lattice = pairs.test_few_pairs_on_a_large_lattice
test_captured_rounds_of_few_large_pairs = pairs.test_captured_rounds_of_few_large_pairs


@pytest.mark.parametrize("level,parent", [(0, lambda k: k), (1, lambda k: k // 2), (3, lambda k: k // 8),
                                          (3, lambda k: np.where(k < 5, 6, 2)), (5, lambda k: (k * 7) % 9),
                                          (7, lambda k: k // 2)])
def test_groups_equal_waves(ctx, flood_torus, level, parent):
    groups.test_groups_equal_waves(ctx, flood_torus, level, parent)


@pytest.mark.parametrize("graph,level", [(False, 5), (True, 8)])
def test_timing_changes_no_path(ctx, graph, level):
    """As many launches with events as without, in every call that has more than one way."""
    m = M.torus(1.0, 0.3, 120, 36, jitter=0.004, seed=9)
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 75)
    tree = ctx.build_tree(lat, level, 0)
    r = ctx.tree_read(tree, level)
    parent = (np.arange(1 << level) // 2).astype(np.int32)
    seen = []
    for mode in (ctx.profile_times, lambda: ctx.profile_enable(0)):
        layer = ctx.layer_init(lat, r["assign"], parent, r["frames"])
        out = []
        mode()
        for call in (lambda: ctx.outer_volume(lat, r["boxes"][:5]), lambda: ctx.outer_volume_q(lat, r["qboxes"][:5]),
                     lambda: ctx.lloyd_step(layer, rounds=16, refit=1, graph=graph),
                     lambda: ctx.lloyd_step(layer, rounds=16, refit=1, graph=graph),
                     lambda: ctx.flood_partition(layer, mode=0)):
            n0 = ctx.profile_read()["launches"]
            got = call()
            out.append((ctx.profile_read()["launches"] - n0, got if isinstance(got, dict) else np.asarray(got).tolist()))
        seen.append((out, ctx.profile_read()["count_launches"], ctx.layer_read(layer)["assign"].tolist()))
        layer.free()
    assert seen[0][0] == seen[1][0] and seen[0][2] == seen[1][2]
    assert seen[0][1] >= 2 and seen[1][1] == 0       # the two counts' launches are timed
    for x in (tree, lat, mesh):
        x.free()


def test_timing_captures_no_new_graph(ctx):
    """A captured iteration is the same graph with profiling on or off, in either mode."""
    m = M.torus(1.0, 0.3, 60, 24, jitter=0.004, seed=11)
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 64)
    tree = ctx.build_tree(lat, 8, 0)
    r = ctx.tree_read(tree, 8)
    parent = (np.arange(256) // 2).astype(np.int32)
    seen = []
    for mode in (lambda: ctx.profile_enable(0), ctx.profile_times, lambda: ctx.profile_enable(1)):
        layer = ctx.layer_init(lat, r["assign"], parent, r["frames"])
        mode()
        n0 = ctx.profile_read()["launches"]
        st = [ctx.lloyd_step(layer, rounds=16, refit=1, graph=True) for _ in range(2)]
        seen.append((st, ctx.profile_read()["launches"] - n0))
        ctx.profile_enable(0)
        layer.free()
    assert seen[0] == seen[1] == seen[2]
    for x in (tree, lat, mesh):
        x.free()
