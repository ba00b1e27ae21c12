"""The pinned host memory of the solvers belongs to the ops object (GPU).

A child process solves, frees everything, resets its own device context, and then owns 64
pinned buffers of the size the solvers use; a solve on a new ops object must not write to
them.  (A slot kept in the process beyond the reset was written to again at its old address,
which by then was the first of these buffers.)
"""
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes as C
import glob
import numpy as np
from paper_0707_0159_gb300 import dmrg2d as D, synth

rt = C.CDLL(sorted(glob.glob("/usr/local/cuda/lib64/libcudart.so*"))[0])
mdl, left, right, _ = synth.workload_ladder2_heisenberg_m64()


def solve():
    ops = D.build_ops(mdl, left, right, stream=0)
    v, p = synth.start_vector(ops.info["n_vec"], 2), C.c_void_p()
    assert rt.cudaMalloc(C.byref(p), C.c_size_t(v.nbytes)) == 0
    assert rt.cudaMemcpy(p, v.ctypes.data_as(C.c_void_p), C.c_size_t(v.nbytes), 1) == 0
    so = D.SolverOpts(**{**D.default_solver_opts(), "max_iter": 20, "krylov_dim": 20,
                         "fixed_steps": 1})
    e, st = C.c_double(), D.SolverStats()
    assert D.lib().dmrg2d_lanczos_ground(ops.ptr, C.byref(so), p, C.byref(e), C.byref(st),
                                         C.c_void_p(0)) == 0
    ops.free()
    assert rt.cudaFree(p) == 0
    return e.value


e0 = solve()
assert rt.cudaDeviceReset() == 0
bufs = []
for _ in range(64):
    q = C.c_void_p()
    assert rt.cudaHostAlloc(C.byref(q), C.c_size_t(512), 0) == 0
    a = np.ctypeslib.as_array(C.cast(q, C.POINTER(C.c_double)), (64,))
    a[:] = 7.0
    bufs.append(a)
assert abs(solve() - e0) <= 1e-12 * abs(e0)
assert all(np.all(a == 7.0) for a in bufs), "a caller's pinned buffer was written to"
print("ok")
"""


def test_no_slot_outlives_its_ops():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-2000:]
