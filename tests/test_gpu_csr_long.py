"""The CSR product of as many entries as an int32 row pointer counts: what the last rows read ahead lies
beyond 2^31 - 1."""
from __future__ import annotations

import pytest

import paper_2606_02887_gb300.snmf as S

pytestmark = pytest.mark.gpu


def test_csr_product_of_2_31_entries():
    import torch
    dev, n, per = "cuda:0", 1 << 20, 2048
    nnz = n * per - 1  # row i: `per` entries, one each in the columns per i, per i + 1, ... modulo n; the last row one fewer
    cols = torch.arange(nnz, dtype=torch.int32, device=dev).remainder_(n)
    vals = torch.ones(nnz, device=dev)
    rp = (torch.arange(n + 1, dtype=torch.int64, device=dev) * per).clamp_max_(nnz).int()
    X = torch.randint(0, 8, (n, 1), device=dev).float()  # whole numbers: the sums are exact
    Y = torch.empty_like(X)
    h = S.snmf_create(S.csr_matrix(n, rp, cols, vals), 1, S.snmf_default_options(precision=S.SNMF_F32))
    try:
        S.snmf_apply(h, X, Y, 1)
    finally:
        S.snmf_destroy(h)
    want = X.view(n // per, per).sum(1).repeat(per)[:, None]
    want[-1] -= X[-1]
    assert torch.equal(Y, want)
