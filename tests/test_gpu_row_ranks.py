"""The row kernels of a step between 64 and 128 columns with a graph term, in FP64 and FP32, against
the oracle; bars of the iterate tests (FP64) and of one step's rounding (FP32, tests of tile edges)."""
import math

import numpy as np
import pytest

import oracle as O
import paper_2606_02887_gb300.snmf as S
from workloads import planted_dense, uniform_init

from gpu_helpers import gpu_solve, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r", [(150, 65), (301, 100), (260, 127), (333, 128)])
def test_graph_step_above_64_columns(n, r):
    A, _ = planted_dense(n, 20, 0.02, seed=n)
    W0 = uniform_init(n, r, math.sqrt(A.mean() / r), seed=n + 1)
    gamma = 0.2 * float(np.linalg.norm(A)) / n
    opts = O.Options(max_iter=1, inner_iters=1, tol=0.0, gamma=gamma, memory=10, objective="closed")
    Wo, Ho, _ = O.snmpbb_penalty(A, W0, W0, opts, L=O.paper_laplacian(A))
    for precision, bar in ((S.SNMF_F64, 1e-10), (S.SNMF_F32, 16 * 2.0 ** -24 * (math.sqrt(n) + math.sqrt(r)))):
        W, H, _, _, _ = gpu_solve(A, W0, r, W0, L="paper", gamma=gamma, max_iter=1, inner_iters=1, tol=0.0,
                                  precision=precision)
        assert rel(W, Wo) <= bar and rel(H, Ho) <= bar
