"""A cluster's frame comes out of either kernel with the same bits whatever the
compiler fuses: the library with lloyd.cu compiled without any contraction of
products and sums, a layer of few clusters against one of many."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import sys
import numpy as np
import paper_2203_10521_gb300 as P
from synth import meshes as M
P.LIB_PATH = sys.argv[1]
ctx = P.Context(0)
m = M.torus(1.0, 0.3, 200, 100, jitter=0.004, seed=5)
mesh = ctx.mesh_create(m.verts, m.tris)
lat = ctx.build_occupancy(mesh, 64)
T, shared = len(m.tris), 997
few = np.minimum(np.arange(T) * 2000 // T, 1999)
few = np.random.default_rng(1).permutation(few)
many = few.copy()
rest = few >= shared
many[rest] = shared + np.arange(rest.sum()) % (20000 - shared)
out = []
for a in (few, many):
    K = int(a.max()) + 1
    out.append(ctx.layer_read(ctx.layer_init(lat, a.astype(np.int32), np.zeros(K, np.int32))))
print(int((out[0]["frames"][:shared] != out[1]["frames"][:shared]).sum()))
"""


def test_frames_do_not_depend_on_what_the_compiler_fuses(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_10521_gb300 import build as B
    B.build()
    objs = [os.path.join(B.OUT, u.replace(".cu", ".o")) for u in B.UNITS]
    plain = str(tmp_path / "lloyd.o")
    objs[B.UNITS.index("lloyd.cu")] = plain
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "--fmad=false", "-c", os.path.join(B.SRC, "lloyd.cu"), "-o", plain],
                   check=True)
    lib = str(tmp_path / "libobbvar_plain.so")
    subprocess.run([B.nvcc(), *B.ARCH, "-shared", "-o", lib, *objs], check=True)
    r = subprocess.run([sys.executable, "-c", SCRIPT, lib], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert int(r.stdout) == 0
