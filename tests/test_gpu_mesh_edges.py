"""Mesh validation by bucketed half-edges against a dictionary of edges: closed
meshes of every shape (fans around one vertex, scattered indices), and broken
ones, with the edge and count that the error names."""
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


def _bipyramid(n):
    a = 2 * np.pi * np.arange(n) / n
    v = np.concatenate([np.stack([np.cos(a), np.sin(a), 0 * a], 1), [[0, 0, 1], [0, 0, -1]]]).astype(np.float32)
    i, j = np.arange(n), (np.arange(n) + 1) % n
    return v, np.concatenate([np.stack([i, j, 0 * i + n], 1), np.stack([j, i, 0 * i + n + 1], 1)]).astype(np.int32)


def _mesh(name):
    if name == "cube":
        m = M.cube()
    elif name == "torus":
        m = M.torus(1.0, 0.3, 40, 21, jitter=0.01, seed=2)
    else:
        return _bipyramid(int(name))
    perm = np.random.Generator(np.random.PCG64(4)).permutation(len(m.verts)).astype(np.int32)
    v = np.empty_like(m.verts)
    v[perm] = m.verts
    return v, perm[m.tris]


def _edges(f):
    e = {}
    for t in f:
        for a, b in ((t[0], t[1]), (t[1], t[2]), (t[2], t[0])):
            k = (min(a, b), max(a, b))
            e[k] = e.get(k, 0) + 1
    return e


@pytest.mark.parametrize("name", ["cube", "torus", "3", "700", "20000"])
def test_closed_meshes(ctx, name):
    v, f = _mesh(name)
    mesh = ctx.mesh_create(v, f)
    # the adjacency through the layer moves it allows: one cluster a triangle half, moves only across edges
    lat = ctx.build_occupancy(mesh, 33)
    assert lat.bits().sum() > 0
    lat.free()
    mesh.free()


@pytest.mark.parametrize("name", ["cube", "torus", "700"])
@pytest.mark.parametrize("damage", ["drop", "repeat", "rewire"])
def test_broken_meshes_name_the_smallest_bad_edge(ctx, name, damage):
    import paper_2203_10521_gb300 as P
    v, f = _mesh(name)
    f = f.copy()
    if damage == "drop":
        f = np.delete(f, len(f) // 2, 0)
    elif damage == "repeat":
        f = np.concatenate([f, f[[5, 5]]])
    else:
        f[3, 1] = next(x for x in range(len(v)) if x not in f[3])
    bad = sorted(k for k, n in _edges(f).items() if n != 2)[0]
    with pytest.raises(P.ObbError) as e:
        ctx.mesh_create(v, f)
    assert e.value.code == -2
    assert f"edge ({bad[0]}, {bad[1]}) is shared by {_edges(f)[bad]} triangles" in str(e.value)


def test_bad_input_codes(ctx):
    import paper_2203_10521_gb300 as P
    v, f = _mesh("torus")
    for what, code in ((("v", np.nan), -1), (("i", len(v)), -1), (("i", -1), -1), (("r", 0), -2)):
        vv, ff = v.copy(), f.copy()
        if what[0] == "v":
            vv[-1, 2] = what[1]
        elif what[0] == "i":
            ff[-1, 1] = what[1]
        else:
            ff[7, 1] = ff[7, 0]
        with pytest.raises(P.ObbError) as e:
            ctx.mesh_create(vv, ff)
        assert e.value.code == code, what


@pytest.mark.parametrize("n", [1, 31, 97, 129, 300, 640, 641, 1025])
def test_counting_copy_and_ranks_of_ragged_lattices(ctx, n):
    """Rows of 1 to 9 chunks, and row runs that cross slices: whole-box counts through the counting copy and its
    rank table are the empty points of the exported words."""
    m = M.icosphere(2, radius=1.0)
    mesh = ctx.mesh_create(m.verts, m.tris)
    lat = ctx.build_occupancy(mesh, n)
    half = 0.5 * (m.verts.max(0) - m.verts.min(0)) * 1.2
    box = np.concatenate([0.5 * (m.verts.max(0) + m.verts.min(0)), [1, 0, 0, 0, 1, 0], half]).astype(np.float32)
    tilt = box.copy()
    tilt[3:9] = [np.cos(0.3), np.sin(0.3), 0, -np.sin(0.3), np.cos(0.3), 0]
    tilt[9:12] *= 2
    cnt, pts = ctx.outer_volume(lat, np.stack([box, tilt]), want_points=True)
    solid = int(lat.bits().sum(dtype=np.int64))
    assert np.array_equal(pts - cnt, [solid, solid])
    lat.free()
    mesh.free()
