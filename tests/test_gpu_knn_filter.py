"""The tensor-core filter of the kNN graph against the unfiltered kernel, bit for bit.

The filter takes up to 128 coordinates; the same points with zero coordinates appended have the same
distances (adding 0 * 0 changes no sum) and go to the unfiltered kernel."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2606_02887_gb300.snmf as S
from workloads import gmm_points

pytestmark = pytest.mark.gpu


def _both(X, k, sr):
    import torch
    X = np.ascontiguousarray(X, dtype=np.float32)
    wide = np.zeros((X.shape[0], 129), dtype=np.float32)
    wide[:, :X.shape[1]] = X
    return [S.snmf_knn_graph(torch.tensor(p, device="cuda:0"), k=k, sigma_rank=sr) for p in (X, wide)]


def _bits(t):
    """The bytes of an output: a similarity that underflows leaves a row of A^ at 0 / 0, a NaN in both."""
    return t.cpu().numpy().tobytes()


@pytest.mark.parametrize("n,d,k", [(1024, 1, 1), (1025, 7, 16), (1087, 32, 17), (2048, 33, 32), (4095, 12, 10),
                                   (4097, 64, 10), (5003, 128, 31), (9001, 8, 5)])
def test_filter_is_exact(n, d, k):
    X, _ = gmm_points(n, d, 5, seed=3 * n + d)
    for a, b in zip(*_both(X, k, min(7, k))):
        assert _bits(a) == _bits(b)


@pytest.mark.parametrize("kind", ["ties", "tight", "copies", "far", "huge"])
def test_filter_hard_points(kind):
    """Rounded points (many equal distances), clusters much tighter than their distance and many copies of
    few points (the filter gives up), points far from the origin, squared distances near overflow."""
    X, lab = gmm_points(3000, 24, 4, seed=9)
    if kind == "ties":
        X = np.round(X)
    elif kind == "tight":
        X = 1e-3 * X + 100.0 * (lab[:, None] % 2)
    elif kind == "copies":
        X = np.repeat(X[:1500], 2, axis=0)
    elif kind == "far":
        X = X + 1000.0
    else:
        X = X * np.float32(1e17)
    for a, b in zip(*_both(X, 9, 7)):
        assert _bits(a) == _bits(b)


@pytest.mark.parametrize("value", [np.nan, np.inf, 3e19])
def test_filter_rejects_non_finite(value):
    import torch
    X, _ = gmm_points(2000, 16, 4, seed=5)
    X = np.asarray(X, dtype=np.float32)
    X[1234, 5] = value
    with pytest.raises(S.SnmfError):
        S.snmf_knn_graph(torch.tensor(X, device="cuda:0"), k=5, sigma_rank=3)
