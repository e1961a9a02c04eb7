"""Kernels at the edges of their tiles: one outer iteration with one step per block against the
oracle, over ranks and row counts around the widths (16, 32, 64) and chunk lengths of the Gram,
the product tiles and the row kernels, and over several restarts.

Bars.  FP64: 1e-10 relative, as the iterate tests.  FP32: a step computes X - (1 + 1.7) g / rho at
most, and g = X G - B rounds by about 2^-24 (sqrt(n) |B| + sqrt(r) |X G|) with |B| <= rho |X|; the
two blocks, and B and G of the second from the first, add up to at most four such errors:
16 * 2^-24 (sqrt(n) + sqrt(r)).
"""
import math

import numpy as np
import pytest

import oracle as O
import paper_2606_02887_gb300.snmf as S
from workloads import planted_dense, uniform_init

from gpu_helpers import gpu_solve, rel

pytestmark = pytest.mark.gpu

SIZES = [(64, 1, 1), (65, 3, 2), (129, 15, 1), (500, 16, 3), (700, 17, 1), (1100, 20, 2), (333, 31, 1), (1025, 32, 2),
         (900, 33, 1), (2100, 63, 1), (640, 64, 3), (500, 65, 1), (450, 100, 2), (400, 128, 1), (390, 129, 1),
         (300, 256, 1)]


def one_step(n, r, b, precision, A=None, **opt):
    A0, _ = planted_dense(n, min(r, 40), 0.02, seed=50 + n)
    A = A0 if A is None else A(A0)
    starts = [uniform_init(n, r, math.sqrt(A.mean() / r), seed=60 + n + j) for j in range(b)]
    W0 = np.concatenate(starts, 1)
    W, H, _, _, per = gpu_solve(A, W0, r, Ht0=W0, precision=precision, batch=b, inner_iters=1, max_iter=1, tol=0.0,
                                nonmonotone_M=10, **opt)
    err = 0.0
    for j in range(b):
        o = O.Options(memory=10, inner_iters=1, max_iter=1, tol=0.0, objective="closed")
        Wo, Ho, _ = O.snmpbb_penalty(A, starts[j], starts[j], o)
        s = slice(j * r, (j + 1) * r)
        err = max(err, rel(W[:, s], Wo), rel(H[:, s], Ho))
        res = np.linalg.norm(A - Wo @ Ho.T) / np.linalg.norm(A)
        assert abs(per["residual"][j] - res) <= 1e-4 * max(res, 1.0)
    return err


def f32_bar(n, r):
    return 16 * 2.0 ** -24 * (math.sqrt(n) + math.sqrt(r))


@pytest.mark.parametrize("n,r,b", SIZES)
def test_f64_step_at_tile_edges(n, r, b):
    assert one_step(n, r, b, S.SNMF_F64) <= 1e-10


@pytest.mark.parametrize("n,r,b", SIZES)
def test_f32_step_at_tile_edges(n, r, b):
    assert one_step(n, r, b, S.SNMF_F32) <= f32_bar(n, r)


@pytest.mark.parametrize("precision,sym", [(S.SNMF_F32, 0), (S.SNMF_BF16, 0), (S.SNMF_BF16, 1), (S.SNMF_FP8, 0)])
@pytest.mark.parametrize("n,r,b", [(64, 2, 1), (127, 16, 1), (130, 17, 1), (259, 33, 1), (300, 5, 13), (1000, 40, 2),
                                   (515, 43, 3)])
def test_final_evaluation_at_tile_edges(n, r, b, precision, sym):
    """The residual of a stored A (FP32, BF16 full and upper tiles, E4M3) from the CUDA-core product
    of the final evaluation, against the factors that the solve returns: entries k / 8 below 2 are
    exact in BF16 and E4M3, so every storage holds the same A.  Bar: the FP32 sums of length n and r,
    2^-24 (sqrt(n) + sqrt(r)) of ||A||^2, on the squared residual."""
    q = np.random.default_rng(n + r)
    A = q.integers(0, 16, (n, n)) / 8.0
    A = np.triu(A) + np.triu(A, 1).T
    W0 = uniform_init(n, r * b, math.sqrt(A.mean() / r), seed=3)
    W, H, _, _, per = gpu_solve(A, W0, r, Ht0=W0, precision=precision, batch=b, sym_half=sym, inner_iters=1, max_iter=1,
                                tol=0.0)
    for j in range(b):
        s = slice(j * r, (j + 1) * r)
        true = (np.linalg.norm(A - W[:, s] @ H[:, s].T) / np.linalg.norm(A)) ** 2
        assert abs(per["residual"][j] ** 2 - true) <= 2.0 ** -24 * (math.sqrt(n) + math.sqrt(r))


def test_batch_of_every_tile_width():
    """The grouped Gram and CUDA-core product of the uneven batch over every tile width, with blocks
    that start off 16 bytes: each problem's step against the oracle."""
    import torch
    ns, rs = [70, 129, 128, 300, 500, 65, 257], [3, 16, 17, 32, 33, 64, 20]
    As = [planted_dense(n, r, 0.02, seed=n)[0] for n, r in zip(ns, rs)]
    Ws = [uniform_init(n, r, math.sqrt(A.mean() / r), seed=n + 1) for n, r, A in zip(ns, rs, As)]
    for prec, dt in ((S.SNMF_F64, torch.float64), (S.SNMF_F32, torch.float32)):
        vals = torch.tensor(np.concatenate([A.ravel() for A in As]), dtype=dt, device="cuda")
        W = torch.tensor(np.concatenate([w.ravel() for w in Ws]), dtype=dt, device="cuda")
        H = W.clone()
        o = S.snmf_default_options(precision=prec, inner_iters=1, max_iter=1, tol=0.0)
        h = S.snmf_create(S.dense_batch_matrix(vals, ns, rs), 0, o)
        S.snmf_solve(h, W, H)
        per = S.snmf_restart_stats(h, len(ns))
        S.snmf_destroy(h)
        W, H, at = W.cpu().double().numpy(), H.cpu().double().numpy(), 0
        for p, (n, r) in enumerate(zip(ns, rs)):
            opt = O.Options(memory=10, inner_iters=1, max_iter=1, tol=0.0, objective="closed")
            Wo, Ho, _ = O.snmpbb_penalty(As[p], Ws[p], Ws[p], opt)
            w, hh = W[at:at + n * r].reshape(n, r), H[at:at + n * r].reshape(n, r)
            at += n * r
            bar = 1e-10 if prec == S.SNMF_F64 else f32_bar(n, r)
            assert rel(w, Wo) <= bar and rel(hh, Ho) <= bar
            true = (np.linalg.norm(As[p] - w @ hh.T) / np.linalg.norm(As[p])) ** 2
            assert abs(per["residual"][p] ** 2 - true) <= 2.0 ** -24 * (math.sqrt(n) + math.sqrt(r))
