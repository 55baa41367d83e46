"""Chi-square joins and top-k on features of any scale and on near-duplicates, against the oracle.

The FP32 distances' absolute error follows the features' largest magnitude, so rows that sum to 1e-15
are told apart as those that sum to 1 are, and so are rows that differ by 1e-6 of their sum: the join
sends as few pairs to FP64, and the top-k ranks more such rows than its lists hold.
"""

import numpy as np
import pytest

import oracle
from paper_1812_07607_gb300 import workloads as W
from test_gpu_hist_topk import _store, check, dl, orc  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu
SCALES = [2.0 ** 39, 1.0, 1e-12, 1e-15, 1e-30, 2.0 ** -126]


@pytest.mark.parametrize("scale", SCALES)
@pytest.mark.parametrize("nQ", [5, 40])   # the few-row path and the tile
def test_topk_small_scales(dl, orc, nQ, scale):
    g = W.rng(9600 + nQ)
    X, _ = W.clustered_histograms(g, 12_000 + nQ, 20, 400, 0.02)
    X = (X * np.float32(scale)).astype(np.float32)
    check(dl, orc, X[:nQ], X[nQ:], 10, "chi2")


@pytest.mark.parametrize("nQ", [5, 40])
def test_topk_near_duplicates(dl, orc, nQ):
    g = W.rng(9610 + nQ)
    X = W.dirichlet_histograms(g, 1, 64) * (1 + 1e-6 * g.random((12_000 + nQ, 64)))
    check(dl, orc, X[:nQ].astype(np.float32), X[nQ:].astype(np.float32), 10, "chi2")


@pytest.mark.parametrize("scale", SCALES)
def test_join_small_scales(dl, orc, scale):
    g = W.rng(9620)
    X, _ = W.clustered_histograms(g, 1500, 32, 100, 0.01)
    X = (X * np.float32(scale)).astype(np.float32)
    R, S = X[:600], X[600:]
    D = np.sort(orc.hist_dist_block(R, S, oracle.METRIC_CHI2).ravel())
    i = len(D) // 200
    i += int(np.argmax(D[i + 1:i + 400] / D[i:i + 399]))   # a threshold between two distances well apart
    t = float(np.sqrt(D[i] * D[i + 1]))
    want = {(int(a), int(b)) for a, b in orc.hist_join(R, S, t, oracle.METRIC_CHI2, oracle.MODE_RXS).tolist()}
    assert D[i + 1] / D[i] > 1 + 1e-4 and want
    for prec in ("auto", "fp32_plain"):
        res = dl.sim_join(_store(dl, np.arange(600), R), _store(dl, np.arange(900), S), t, metric="chi2", precision=prec)
        a, b = res.pairs_host()
        band = res.stats()["band_pairs"]
        res.free()
        assert set(zip(a.tolist(), b.tolist())) == want and len(a) == len(want), prec
        assert band <= 2   # nothing within (d + 16) 2^-23 of t but what lies next to it
