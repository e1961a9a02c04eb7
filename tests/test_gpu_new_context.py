"""The allocation-free product and the kNN graph after a device reset: a context in which no kernel has been
launched yet.  In a process of its own, which holds nothing else on the device."""
from __future__ import annotations

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import ctypes as C
import numpy as np
import paper_2606_02887_gb300.snmf as S
lib = S.load_library()
rt = lib  # names are looked up in the runtime that the library is linked with as well
rt.cudaMalloc.argtypes = [C.POINTER(C.c_void_p), C.c_size_t]
rt.cudaMemcpy.argtypes = [C.c_void_p, C.c_void_p, C.c_size_t, C.c_int]
def up(a):
    p = C.c_void_p()
    assert rt.cudaMalloc(C.byref(p), a.nbytes) == 0 and rt.cudaMemcpy(p, a.ctypes.data, a.nbytes, 1) == 0
    return p
def down(p, a):
    assert rt.cudaMemcpy(a.ctypes.data, p, a.nbytes, 2) == 0
    return a
rng = np.random.default_rng(3)
n, cols, m, k = 2048, 64, 1500, 8
A, X = rng.integers(0, 8, (n, n)), rng.integers(0, 8, (n, cols))  # whole numbers: every sum is exact
P = rng.standard_normal((m, 100)).astype(np.float32)
def calls():
    out = []
    for dt, code in ((np.float32, S.SNMF_F32), (np.float64, S.SNMF_F64)):
        Y, x = np.zeros((n, cols), dt), C.c_double()
        y = up(Y)
        assert lib.snmf_apply_dense_noalloc(up(A.astype(dt)), code, n, n, up(X.astype(dt)), y, cols, C.byref(x), None) == 0
        assert (down(y, Y) == A @ X).all()
    i, f, nnz = np.zeros(2 * m * k, np.int32), np.zeros(2 * m * k, np.float32), C.c_int64()
    rp, ci, ah = up(np.zeros(m + 1, np.int32)), up(i), up(f)
    assert lib.snmf_knn_graph(up(P), m, 100, k, 7, rp, ci, ah, None, None, 2 * m * k, C.byref(nnz), None) == 0
    return [nnz.value, down(ci, i)[:nnz.value].tobytes(), down(ah, f)[:nnz.value].tobytes()]
first = calls()
assert rt.cudaDeviceReset() == 0
assert calls() == first
print("as before")
"""


def test_calls_after_a_device_reset():
    p = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT), capture_output=True,
                       text=True, timeout=300)
    assert p.returncode == 0 and p.stdout.strip().endswith("as before"), p.stderr[-2000:]
