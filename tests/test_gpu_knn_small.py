"""The kNN filter where squared distances come near the smallest normal number or below it: products and
norms are then rounded absolutely, which its relative bounds do not cover."""
from __future__ import annotations

import numpy as np
import pytest

from test_gpu_knn_filter import _bits, _both
from workloads import gmm_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-17, 1e-19, 1e-20, 1e-21, 1e-22, 5e-23])
@pytest.mark.parametrize("kind", ["all", "half"])
def test_filter_small_points(kind, scale):
    """Points scaled down, all of them or every other one (those lie at one place for the rest)."""
    X, _ = gmm_points(3000, 24, 4, seed=9)
    X = np.asarray(X, dtype=np.float32)
    if kind == "all":
        X *= np.float32(scale)
    else:
        X[::2] *= np.float32(scale)
    for a, b in zip(*_both(X, 9, 7)):
        assert _bits(a) == _bits(b)
