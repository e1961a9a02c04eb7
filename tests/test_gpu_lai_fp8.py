"""The eigen-sketch of an A in E4M3 codes: its products see the stored values, as those of the same values in FP32
do, in the same order, so the starts made of the two sketches are the same bits."""
from __future__ import annotations

import numpy as np
import pytest

import oracle.fp8 as F8
import paper_2606_02887_gb300.snmf as S
from workloads import planted_dense

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r", [(300, 6), (389, 40)])
def test_sketch_of_fp8_codes(n, r):
    import torch
    A, _ = planted_dense(n, 6, 0.05, seed=n)
    A = np.asarray(A, dtype=np.float32)
    stored = F8.quantize(A)[2]
    W = []
    for M, precision in ((A, S.SNMF_FP8), (stored, S.SNMF_F32)):
        h = S.snmf_create(S.dense_matrix(torch.tensor(M, dtype=torch.float32, device="cuda:0")), r,
                          S.snmf_default_options(precision=precision))
        try:
            w = torch.zeros(n, r, device="cuda:0")
            S.snmf_svd_init(h, w, None, 10, 2, 5)
        finally:
            S.snmf_destroy(h)
        W.append(w.cpu().numpy())
    assert np.isfinite(W[0]).all() and np.array_equal(W[0], W[1])
