"""The histogram top-k against stores of a few rows, whose distances the selecting kernel forms itself.

Bit-exact against the oracle on both sides of that line (128 rows, 200 for up to 256 query rows), for few and many query rows, feature
counts with and without whole quads, and k below, at and above the store's size; one kernel each up to
the line.
"""

import numpy as np
import pytest

from paper_1812_07607_gb300 import workloads as W
from test_gpu_hist_topk import _store, check, dl, orc  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("metric", ["l1", "chi2"])
@pytest.mark.parametrize("nS", [1, 2, 31, 127, 128, 129, 200, 201])
@pytest.mark.parametrize("nQ,d,k", [(1, 5, 1), (40, 64, 10), (700, 18, 128), (3, 260, 200)])
def test_exact(dl, orc, metric, nS, nQ, d, k):
    g = W.rng(9900 + nS + nQ)
    X, _ = W.clustered_histograms(g, nQ + nS, d, 12, 0.02)
    check(dl, orc, X[:nQ], X[nQ:], k, metric)


@pytest.mark.parametrize("metric", ["l1", "chi2"])
def test_one_kernel(dl, metric):
    X = W.dirichlet_histograms(W.rng(9950), 400, 24)
    for nQ, nS, kernels in ((300, 128, 1), (300, 129, 2), (256, 200, 1), (256, 201, 2), (257, 200, 2)):
        res = dl.topk_join(_store(dl, np.arange(nQ), X[:nQ]), _store(dl, np.arange(nS), X[:nS]), 5, metric=metric)
        assert res.stats()["kernels_launched"] == kernels
        res.free()
