"""A graph-regularised solve of more rows than 64 x 65535, the most that a grid whose rows of tiles lie on
its second index holds.  Most rows belong to nodes without edges that start at zero, where they stay, so
the others follow the small problem that they make up."""
from __future__ import annotations

import numpy as np
import pytest

import oracle as O
import paper_2606_02887_gb300.snmf as S
from gpu_helpers import rel
from test_gpu_parity import ITER_TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [2, 3])  # rows of 16 bytes, and not
def test_graph_solve_of_many_rows_fp64(r):
    import torch
    m, n, lam, gamma = 600, 64 * 65536 + 2, 0.3, 0.1
    at = 6991 * np.arange(m)  # the parity of the small problem's row, which the start of ||L||_2 depends on
    at[-1] = n - 1
    rng = np.random.default_rng(11)
    A = np.triu(rng.random((m, m)) * (rng.random((m, m)) < 0.02), 1)
    A += A.T
    L = np.diag(A.sum(1)) - A
    W0 = rng.random((m, r))
    Wo, Ho, _ = O.snmpbb_penalty(A, W0, W0, O.Options(lambda_sym=lam, max_iter=3, tol=0.0, gamma=gamma, memory=10,
                                                      objective="closed"), L=L)

    def csr(M):
        i, j = np.nonzero(M)
        rp = np.zeros(n + 1, dtype=np.int64)
        rp[1 + at] = np.bincount(i, minlength=m)
        return (torch.tensor(np.cumsum(rp), dtype=torch.int32, device="cuda:0"),
                torch.tensor(at[j], dtype=torch.int32, device="cuda:0"), torch.tensor(M[i, j], device="cuda:0"))

    W = torch.zeros(n, r, dtype=torch.float64, device="cuda:0")
    W[torch.tensor(at, device="cuda:0")] = torch.tensor(W0, device="cuda:0")
    H = W.clone()
    a, l = csr(A), csr(L)
    h = S.snmf_create(S.csr_matrix(n, *a), r, S.snmf_default_options(precision=S.SNMF_F64, lambda_sym=lam, max_iter=3, tol=0.0))
    try:
        S.snmf_set_graph_reg(h, S.csr_matrix(n, *l), gamma)
        S.snmf_solve(h, W, H)
    finally:
        S.snmf_destroy(h)
    W, H = W.cpu().numpy(), H.cpu().numpy()
    assert rel(W[at], Wo) <= ITER_TOL and rel(H[at], Ho) <= ITER_TOL
    W[at], H[at] = 0.0, 0.0
    assert not W.any() and not H.any()
