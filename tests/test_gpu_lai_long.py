"""The low-rank product of long factors: a CTA that walks several row tiles (16-byte rows) against the
kernel of one tile per CTA, which an odd number of columns takes, on the same sketch.

Bar: both sum 64 products in FP32 in one order, from U^T X whose sums over n may be split differently:
2^-24 (sqrt(n) + 8) of the largest entry."""
from __future__ import annotations

import math

import numpy as np
import pytest

import paper_2606_02887_gb300.snmf as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cols", [(130001, 32), (117000, 16), (125003, 64), (140100, 48)])
def test_product_of_long_factors(n, cols):
    import torch
    rng = np.random.default_rng(n)
    v = rng.random(n - 1).astype(np.float32)
    d = (1.0 + rng.random(n)).astype(np.float32)
    rows = np.concatenate([np.arange(n), np.arange(n - 1), np.arange(1, n)])
    cidx = np.concatenate([np.arange(n), np.arange(1, n), np.arange(n - 1)])
    vals = np.concatenate([d, v, v])
    order = np.lexsort((cidx, rows))
    rp = np.zeros(n + 1, dtype=np.int32)
    np.cumsum(np.bincount(rows, minlength=n), out=rp[1:])
    csr = [torch.tensor(a, device="cuda:0") for a in (rp, cidx[order].astype(np.int32), vals[order])]
    X = torch.rand(n, cols, generator=torch.Generator().manual_seed(7)).to("cuda:0")
    out = []
    for r in (cols, cols - 1):
        h = S.snmf_create(S.csr_matrix(n, *csr), r, S.snmf_default_options(precision=S.SNMF_F32))
        try:
            S.snmf_lai_sketch(h, 64, 10, 1, 99)
            Y = torch.empty(n, r, device="cuda:0")
            S.snmf_apply(h, X[:, :r].contiguous(), Y, r)
            out.append(Y[:, :cols - 1].double())
        finally:
            S.snmf_destroy(h)
    bar = 2.0 ** -24 * (math.sqrt(n) + 8) * float(out[1].abs().max())
    assert float((out[0] - out[1]).abs().max()) <= bar
