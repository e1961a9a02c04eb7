"""What the library asks of the CUDA runtime, on the CPU: the calls run in a process of their own with a
stand-in for the runtime (tests/fake/cudart.c) that checks every launch against the limits of a device
and of its context, and refuses what a test tells it to."""
from __future__ import annotations

import json
import os
import shutil
import subprocess
import sys

import pytest

import paper_2606_02887_gb300.snmf as S

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA_INCLUDE = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

PRELUDE = """
import ctypes as C, json, sys
import numpy as np
import paper_2606_02887_gb300.snmf as S
fake = C.CDLL(None)
fake.fake_log.restype = C.c_char_p
fake.fake_memory.argtypes = [C.c_size_t]
def log():  # [code, device, kernel, grid, threads, dynamic shared memory] of every launch since fake_clear()
    out = []
    for l in fake.fake_log().decode().splitlines():
        w = l.split()
        if w[0] != "alloc":
            out.append([int(w[0]), int(w[1]), w[2], [int(x) for x in w[3:6]], int(w[6]), int(w[7])])
    return out
def ring(n, dtype=np.float32):  # CSR of a cycle
    i = np.arange(n)
    cols = np.sort(np.stack([(i - 1) % n, (i + 1) % n], 1), 1)
    return np.arange(0, 2 * n + 1, 2, dtype=np.int32), cols.reshape(-1).astype(np.int32), np.ones(2 * n, dtype)
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    if not shutil.which("gcc") or not os.path.exists(os.path.join(CUDA_INCLUDE, "cuda_runtime_api.h")):
        pytest.skip("no compiler or CUDA headers")
    if not os.path.exists(S.LIB_PATH):
        from paper_2606_02887_gb300.build import build_library
        build_library()
    so = str(tmp_path_factory.mktemp("fake") / "cudart.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-I" + CUDA_INCLUDE, os.path.join(HERE, "fake", "cudart.c"), "-o", so],
                   check=True)

    def run(script):
        """The JSON that `script` prints in a process on the stand-in."""
        env = dict(os.environ, LD_PRELOAD=so, PYTHONPATH=ROOT)
        p = subprocess.run([sys.executable, "-c", PRELUDE + script], env=env, cwd=ROOT, capture_output=True, text=True,
                           timeout=600)
        assert p.returncode == 0, p.stderr[-2000:]
        return json.loads(p.stdout.strip().splitlines()[-1])

    return run


def test_graph_solve_of_many_rows(fake):
    """Every launch of a graph-regularised solve of n = 4194305 rows is one that the device takes (grid.y and
    grid.z end at 65535: 64 rows each in k_xnext)."""
    got = fake("""
n = 64 * 65536 + 1
A = ring(n)
h = S.snmf_create(S.csr_matrix(n, *A), 1, S.snmf_default_options(max_iter=1, inner_iters=1))
S.snmf_set_graph_reg(h, S.csr_matrix(n, *A), 0.1)
W = np.ones((n, 1), np.float32)
try:
    st = S.snmf_solve_host(h, W, W.copy())[0]
except S.SnmfError as e:
    st = str(e)
print(json.dumps([st, [l for l in log() if l[0]], sum("k_xnext" in l[2] for l in log())]))
""")
    assert got[1] == [] and got[2] > 0 and got[0] == S.SNMF_OK


@pytest.mark.parametrize("kind,kernel", [("csr", "k_rowstep"), ("csr", "k_ctl_final_pen"), ("direct", "k_xupd"),
                                         ("bf16", "k_gemm_tc"), ("batch", "k_bfinal"), ("batch", "k_brow")])
def test_refused_launch_is_not_recorded(fake, kind, kernel):
    """A solve whose launch is refused while its iteration is recorded fails, and the next one on the handle
    launches that kernel again instead of replaying the rest."""
    first, again, state = fake(f"""
kind, kernel = {kind!r}, {kernel!r}
n, r = 320, 4
o = dict(max_iter=1, inner_iters=2)
if kind == "csr":
    h = S.snmf_create(S.csr_matrix(n, *ring(n)), r, S.snmf_default_options(**o))
elif kind == "batch":
    h = S.snmf_create(S.dense_batch_matrix(np.ones(2 * n * n, np.float32), [n, n], [r, r]), 0, S.snmf_default_options(**o))
else:
    if kind == "direct":
        o["formulation"] = S.SNMF_DIRECT
    else:
        o["precision"] = S.SNMF_BF16
    h = S.snmf_create(S.dense_matrix(np.ones((n, n), np.float32)), r, S.snmf_default_options(**o))
W = np.ones(2 * n * r if kind == "batch" else (n, r), np.float32)
out = []
for refuse in (kernel, "none"):
    fake.fake_refuse(refuse.encode())
    fake.fake_clear()
    try:
        S.snmf_solve_host(h, W, None if kind == "direct" else W.copy())
        out.append("solved")
    except S.SnmfError as e:
        out.append("failed")
out.append([l[0] for l in log() if kernel in l[2]])
print(json.dumps(out))
""")
    assert first == "failed" and again == "solved" and state and not any(state)
