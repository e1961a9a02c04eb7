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


@pytest.mark.parametrize("kind", ["noalloc_f32", "noalloc_f64", "knn", "f32_r200", "f64", "direct", "bf16", "fp8", "lai",
                                  "batch"])
def test_shared_memory_limit_of_each_context(fake, kind):
    """The dynamic shared memory above 48 KB that a kernel is launched with has been allowed in the context of
    the launch: on the first device, on another one, and after a device reset."""
    codes, most = fake(f"""
kind = {kind!r}
def call():
    if kind.startswith("noalloc"):
        t = np.float64 if kind.endswith("64") else np.float32
        A, X, Y, x = np.ones((2048, 2048), t), np.ones((2048, 64), t), np.ones((2048, 64), t), C.c_double()
        p = lambda a: a.ctypes.data_as(C.c_void_p)
        return S.load_library().snmf_apply_dense_noalloc(p(A), S.SNMF_F64 if t is np.float64 else S.SNMF_F32, 2048, 2048,
                                                         p(X), p(Y), 64, C.byref(x), None)
    if kind == "knn":
        n, k = 1500, 8
        X, i, f, nnz = np.ones((n, 100), np.float32), np.zeros(2 * n * k, np.int32), np.zeros(2 * n * k, np.float32), C.c_int64()
        p = lambda a: a.ctypes.data_as(C.c_void_p)
        rp = np.zeros(n + 1, np.int32)
        return S.load_library().snmf_knn_graph(p(X), C.c_int64(n), 100, k, 7, p(rp), p(i), p(f), None, None,
                                               C.c_int64(2 * n * k), C.byref(nnz), None)
    n, r, o = 1024, 40, dict(max_iter=1, inner_iters=1, batch=2)
    if kind == "f32_r200":
        r = 200
    elif kind == "f64":
        r, o["precision"] = 100, S.SNMF_F64
    elif kind == "direct":
        n, r, o["formulation"] = 4096, 64, S.SNMF_DIRECT
    elif kind in ("bf16", "fp8"):
        r, o["precision"] = 64, S.SNMF_BF16 if kind == "bf16" else S.SNMF_FP8
    if kind == "batch":
        A = S.dense_batch_matrix(np.ones(2 * n * n, np.float32), [n, n], [10, 60])
        r, o["batch"] = 0, 1
    elif kind == "lai":
        A = S.csr_matrix(n, *ring(n))
    else:
        A = S.dense_matrix(np.ones((n, n), np.float64 if kind == "f64" else np.float32))
    h = S.snmf_create(A, r, S.snmf_default_options(**o))
    if kind == "lai":
        S.snmf_lai_sketch(h, 64, 10, 1, 1)
    W = np.ones(n * 70 if kind == "batch" else (n, r * 2), np.float64 if kind == "f64" else np.float32)
    st = S.snmf_solve_host(h, W, None if kind == "direct" else W.copy())[0]
    S.snmf_destroy(h)
    return st
def tried():
    try:
        return call()
    except S.SnmfError as e:
        return str(e)
codes = [tried()]
fake.fake_device(1)
codes.append(tried())
fake.fake_device(0)
codes.append(tried())
fake.fake_reset(0)
codes.append(tried())
print(json.dumps([codes + sorted(set((l[0], l[2][:80]) for l in log() if l[0])), max(l[5] for l in log())]))
""")
    assert all(c == codes[0] and not isinstance(c, str) for c in codes), codes
    assert codes[0] >= 0 or kind == "knn"  # no kernel runs, so the graph of the points holds what it may
    assert most > 48 * 1024


def test_noalloc_scratch_of_each_context(fake):
    """The address of the allocation-free product's scratch is resolved once in a context, and again in the
    one after a device reset, whose handle may have the address of the old one."""
    assert fake("""
def call():
    A, X, Y, x = np.ones((512, 512)), np.ones((512, 8)), np.ones((512, 8)), C.c_double()
    p = lambda a: a.ctypes.data_as(C.c_void_p)
    assert S.load_library().snmf_apply_dense_noalloc(p(A), S.SNMF_F64, 512, 512, p(X), p(Y), 8, C.byref(x), None) == 0
    return fake.fake_symbols()
out = [call(), call()]
fake.fake_reset(0)
out += [call(), call()]
fake.fake_device(1)
print(json.dumps(out + [call(), call()]))
""") == [1, 1, 2, 2, 3, 3]


def test_knn_graph_without_room_for_the_filter(fake):
    """Where the filter's workspace cannot be had, the call runs without the filter instead of failing, and where
    the partial lists cannot be had without those; where nothing can be had, it fails."""
    got = fake("""
n, d, k = 20000, 64, 10
X, i, f = np.ones((n, d), np.float32), np.zeros(2 * n * k, np.int32), np.zeros(2 * n * k, np.float32)
rp, nnz = np.zeros(n + 1, np.int32), C.c_int64()
p = lambda a: a.ctypes.data_as(C.c_void_p)
out = []
for most in (0, 40 << 20, 12 << 20, 1 << 20):
    fake.fake_memory(most)
    fake.fake_clear()
    st = S.load_library().snmf_knn_graph(p(X), n, d, k, 7, p(rp), p(i), p(f), None, None, 2 * n * k, C.byref(nnz), None)
    out.append([st, sum("k_knn_tc" in l[2] for l in log()), sum("5k_knnE" in l[2] for l in log()),
                sum("k_knn_merge" in l[2] for l in log())])
print(json.dumps(out))
""")
    assert [g[0] for g in got] == [S.SNMF_OK] * 3 + [S.SNMF_ERR_OOM]
    assert got[0][1] == 2 and got[1][1:] == [0, 1, 1] and got[2][1:] == [0, 1, 0] and got[3][1:] == [0, 0, 0]


def test_tensor_core_row_kernels_run_block_steps_alone(fake):
    """A tuned handle's TF32 row kernels run the steps of its two blocks and no other: not the gradient of the
    start, and no step of a handle with a graph term, which run in FP32."""
    tuned, with_graph, without = fake("""
n, r = 1024, 64
h = S.snmf_create(S.dense_matrix(np.ones((n, n), np.float32)), r, S.snmf_default_options(max_iter=1, inner_iters=2, autotune=1))
out = []
for gamma in (None, 0.1, 0.0):
    if gamma is not None:
        S.snmf_set_graph_reg(h, S.csr_matrix(n, *ring(n)) if gamma else None, gamma)
    W = np.ones((n, r), np.float32)
    fake.fake_clear()
    S.snmf_solve_host(h, W, W.copy())
    names = [l[2] for l in log()]
    out.append([sum(k in m for m in names) for k in ("k_rowtc_grad", "k_rowtma", "k_rowtc_dstep")])
print(json.dumps(out))
""")
    assert tuned == without and tuned[0] == 2 and tuned[1] + 2 * tuned[2] == 8 and with_graph == [0, 0, 0]


def test_cached_splits_of_other_tiles(fake, tmp_path):
    """A tuning cache's K split of an FP32 product counts for the tiles that it was timed with alone: a cache
    in the first format leaves the split to the built-in rule and keeps the rest, one in the present
    format, or in none that the library writes, counts as it is."""
    plain, got, written = fake(f"""
r = 64
def solve(fmt, n=4096):
    o = dict(max_iter=1, inner_iters=1)
    if fmt is not None:
        path = {str(tmp_path)!r} + f"/{{len(fmt)}}.json"
        if fmt:
            entry = dict(splits=3, row_tc=1, ms=1.0)
            json.dump({{"format": fmt, "devices": {{"fake/152": {{f"dense/f32/n{{n}}/r{{r}}/N{{r}}": entry}}}}}}, open(path, "w"))
        o.update(autotune=1, tune_cache=path)
    h = S.snmf_create(S.dense_matrix(np.ones((n, n), np.float32)), r, S.snmf_default_options(**o))
    W = np.ones((n, r), np.float32)
    fake.fake_clear()
    S.snmf_solve_host(h, W, W.copy())
    # the final evaluation is not tuned
    return [sorted(set(l[3][2] for l in log() if "k_gemm_dense" in l[2])), S.snmf_step_config(h)["body"]]
v = "snmf_gb300 product tuning cache, v"
out = [solve(None)[0], [solve(v + "1"), solve(v + "2"), solve("another")]]
solve("", 2048)  # not in the cache that this process has read
print(json.dumps(out + [json.load(open({str(tmp_path)!r} + "/0.json"))["format"]]))
""")
    assert 3 not in plain and got == [[plain, 3], [[3] + plain, 3], [[3] + plain, 3]]
    assert written == "snmf_gb300 product tuning cache, v2"


@pytest.mark.parametrize("controller", [0, 1])
def test_step_config_with_a_graph_term(fake, controller):
    """snmf_step_config reports the W block's kernels, which a graph term on the H block does not change: the
    recomputing body, 4 and 6 arrays, rows of its own tiles."""
    got = fake(f"""
n, r = 1000, 20
o = S.snmf_default_options(max_iter=1, step_controller={controller}, mlp_weights=True)
w = np.zeros(S.SNMF_MLP_NPARAMS, np.float32)
h = S.snmf_create(S.csr_matrix(n, *ring(n)), r, o, mlp_weights=w if {controller} else None)
out = []
for gamma in (0.0, 0.1):
    S.snmf_set_graph_reg(h, S.csr_matrix(n, *ring(n)) if gamma else None, gamma)
    out.append(S.snmf_step_config(h))
print(json.dumps(out))
""")
    n_bytes = 1000 * 20 * 4
    assert got[0] == got[1] and got[0]["body"] == 2
    assert got[0]["dstep_bytes"] == 4 * n_bytes and got[0]["update_bytes"] == 6 * n_bytes and got[0]["rows_per_cta"] == 12


def test_handle_with_room_for_eight_slices(fake):
    """A dense handle whose device has no room for ten split-K slices takes eight, and is not refused."""
    most, codes = fake("""
n, r = 1024, 256
A, codes, whole = np.ones((n, n), np.float32), [], 0
for less in (0, 1, 3 << 20):  # a factor is 1 MB, and eight slices take 2 MB less than ten
    fake.fake_memory(max(0, whole - less))
    try:
        fake.fake_clear()
        h = S.snmf_create(S.dense_matrix(A), r, S.snmf_default_options(max_iter=1, inner_iters=1))
        whole = whole or max(int(l.split()[1]) for l in fake.fake_log().decode().splitlines() if l.startswith("alloc"))
        W = np.ones((n, r), np.float32)
        fake.fake_clear()
        codes.append(S.snmf_solve_host(h, W, W.copy())[0])
        slices = max(l[3][2] for l in log() if "k_gemm_dense" in l[2])
    except S.SnmfError as e:
        codes.append(e.status)
print(json.dumps([slices, codes]))
""")
    assert codes == [S.SNMF_OK, S.SNMF_OK, S.SNMF_ERR_OOM] and most <= 8


@pytest.mark.parametrize("n,k,precision", [(500, 10, S.SNMF_F32), (700, 64, S.SNMF_F64), (2048, 64, S.SNMF_F32),
                                           (4100, 20, S.SNMF_F64), (12000, 64, S.SNMF_F32)])
def test_sketch_product_keeps_its_order(fake, n, k, precision):
    """K of a dense sketch's products is split by the rule that a seed's eigenpairs go with, whatever the
    product's tiles: powers of two up to 304 CTAs of 64 x 64, 256 columns and four slices of workspace."""
    got = fake(f"""
n, k, precision = {n}, {k}, {precision}
t = np.float64 if precision == S.SNMF_F64 else np.float32
h = S.snmf_create(S.dense_matrix(np.ones((n, n), t)), 4, S.snmf_default_options(precision=precision))
fake.fake_clear()
try:
    S.snmf_lai_sketch(h, k, 10, 2, 1)
except S.SnmfError:
    pass  # nothing runs, so the factorizations see zeros
print(json.dumps([l[3][2] for l in log() if "k_gemm_dense" in l[2]]))
""")
    tiles, sp = -(-(k + 10) // 64) * -(-n // 64), 1
    while tiles * sp < 304 and n // (2 * sp) >= 256:
        sp *= 2
    if sp > 4:
        sp = 1
    assert got == 4 * [-(-n // (-(-(-(-n // sp)) // 16) * 16))]
