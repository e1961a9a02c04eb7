"""snmf_apply on the caller's buffers against its staged form: in place, off 16 bytes, and with fewer
columns than the handle, in every storage of A.  The same kernel runs on the same values, so the results
are the same bits; <X, A X> is checked against the product in FP64."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2606_02887_gb300.snmf as S
from workloads import planted_dense

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [S.SNMF_F64, S.SNMF_F32, S.SNMF_BF16, S.SNMF_FP8])
@pytest.mark.parametrize("n,r,b", [(200, 16, 1), (131, 7, 3), (300, 48, 2)])
def test_apply_forms_agree(n, r, b, precision):
    import torch
    dt = torch.float64 if precision == S.SNMF_F64 else torch.float32
    A, _ = planted_dense(n, 5, 0.02, seed=n)
    Ad = torch.tensor(A, dtype=dt, device="cuda:0")
    N = r * b
    X = torch.rand(n, N, generator=torch.Generator().manual_seed(3), dtype=torch.float64).to(dt).to("cuda:0")
    h = S.snmf_create(S.dense_matrix(Ad), r, S.snmf_default_options(precision=precision, batch=b))
    try:
        Y = torch.empty_like(X)
        dot = S.snmf_apply(h, X, Y, N)
        true = float((X.double() * Y.double()).sum())
        assert abs(dot - true) <= (1e-12 if dt == torch.float64 else 2.0 ** -20) * abs(true)
        Z = X.clone()  # in place
        assert S.snmf_apply(h, Z, Z, N) == dot and torch.equal(Z, Y)
        room = torch.zeros(n * N + 1, dtype=dt, device="cuda:0")  # one value off the alignment
        off = room[1:].view(n, N)
        off.copy_(X)
        W = torch.empty_like(X)
        assert S.snmf_apply(h, off, W, N) == dot and torch.equal(W, Y)
        if N > 4:  # fewer columns: the rest are zeros
            part = torch.empty(n, N - 3, dtype=dt, device="cuda:0")
            S.snmf_apply(h, X[:, :N - 3].contiguous(), part, N - 3)
            assert torch.equal(part, Y[:, :N - 3])
    finally:
        S.snmf_destroy(h)
