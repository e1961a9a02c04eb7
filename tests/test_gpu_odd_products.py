"""Dense products of odd sizes and columns, whose rows start on single values: every tile width, several K
splits, and the finish pass of single values, in zeros and ones, so that every sum is exact."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2606_02887_gb300.snmf as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [S.SNMF_F32, S.SNMF_F64])
@pytest.mark.parametrize("n", [1, 63, 101, 258, 1001, 2003])
def test_products_of_odd_columns(n, precision):
    import torch
    dt = torch.float32 if precision == S.SNMF_F32 else torch.float64
    g = torch.Generator(device="cuda:0").manual_seed(n)
    A = torch.randint(0, 2, (n, n), generator=g, device="cuda:0").to(dt)
    for cols in (1, 3, 9, 13, 17, 33, 65, 127, 129):
        X = torch.randint(0, 2, (n, cols), generator=g, device="cuda:0").to(dt)
        Y = torch.full_like(X, -1.0)
        want = A.cpu().numpy().astype(np.int64) @ X.cpu().numpy().astype(np.int64)
        xax = S.snmf_apply_dense_noalloc(A, X, Y)
        assert np.array_equal(Y.cpu().numpy(), want) and xax == float((X.cpu().numpy() * want).sum())
        if cols > n or cols > 100:
            continue
        h = S.snmf_create(S.dense_matrix(A), cols, S.snmf_default_options(precision=precision))
        try:
            Y.fill_(-1.0)
            xax = S.snmf_apply(h, X, Y, cols)
        finally:
            S.snmf_destroy(h)
        assert np.array_equal(Y.cpu().numpy(), want) and xax == float((X.cpu().numpy() * want).sum())
