"""Rotation descent against the oracle over cluster sizes: single triangles,
one vertex-gathering pass per cluster, several, and clusters whose probes take
a block each."""
import numpy as np
import pytest

import oracle as O
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
def setup(ctx):
    m = M.torus(1.0, 0.3, 96, 48, jitter=0.004, seed=13)     # 9,216 triangles
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, 48)
    P = O.Problem(m.verts, m.tris, 48)
    yield len(m.tris), lat, P
    lat.free()
    mesh.free()


# 9,216, 3,072 and 2,304 triangles a cluster: a block a box; 1,843 to 257: several passes; 256, 255 and fewer: one
@pytest.mark.parametrize("K,shuffled", [(K, False) for K in (1, 3, 4, 5, 17, 35, 36, 37, 2000, 9216)] +
                         [(K, True) for K in (3, 5, 37)])
def test_descent_over_cluster_sizes(ctx, setup, K, shuffled):
    T, lat, P = setup
    assign = (np.arange(T, dtype=np.int64) * K // T).astype(np.int32)
    if shuffled:   # no vertex shared more than by chance
        assign = np.random.default_rng(K).permutation(assign)
    parent = np.arange(K, dtype=np.int32)                    # no siblings: no moves
    frames = O.cluster_frames(P.V, P.F, assign, K, P.center)
    layer = ctx.layer_init(lat, assign, parent, frames)
    L = O.layer_from_frames(P, assign, parent, frames)
    for graph in (False, True):
        st = ctx.lloyd_step(layer, rounds=1, refit=2, descent_steps=3, graph=graph)
        before = L.obv.copy()
        O.lloyd_step(P, L, rounds=1, do_refit=2, descent_steps=3)
        g = ctx.layer_read(layer)
        assert np.array_equal(g["frames"], L.frames)
        assert np.array_equal(g["qboxes"]["n"], L.n) and np.array_equal(g["qboxes"]["b"], L.bnd)
        assert np.array_equal(g["obv"], L.obv)
        assert st["total_obv"] == int(L.obv.sum()) and (st["refits_accepted"] > 0) == bool((L.obv < before).any())
    layer.free()
