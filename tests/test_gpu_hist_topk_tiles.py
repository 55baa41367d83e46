"""The tiled histogram top-k at the edges of its tiles, groups and lists, bit-exact against the oracle.

Query counts on both sides of the few-row path (16 rows for L1, 32 for chi-square) and of the 128-row tile; store sizes around the
128-column tile and the 2,048 column groups whose minima bound a row's k-th distance; k below, at and
above the groups that hold a column; feature counts that are no multiple of 4 or of the 16-wide K
slice; and enough exact ties to pass the list in shared memory (1,024) and the one behind it (8,192).
"""

import numpy as np
import pytest

from paper_1812_07607_gb300 import workloads as W
from test_gpu_hist_topk import _store, check, dl, orc  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("metric", ["l1", "chi2"])
@pytest.mark.parametrize("nQ,nS,d,k", [
    (1, 2049, 128, 1), (16, 2047, 16, 3), (17, 127, 15, 127), (32, 129, 17, 130), (33, 640, 18, 6), (127, 2048, 33, 9),
    (129, 4097, 20, 1024), (26, 700, 1, 5), (3, 1023, 1, 1023), (130, 8191, 12, 300), (40, 40, 1024, 12),
])
def test_edges_exact(dl, orc, metric, nQ, nS, d, k):
    g = W.rng(9300 + nQ + nS + d + k)
    X, _ = W.clustered_histograms(g, nQ + nS, d, 40, 0.02)   # clipped jitter: exact zero bins
    check(dl, orc, X[:nQ], X[nQ:], k, metric)


@pytest.mark.parametrize("metric", ["l1", "chi2"])
@pytest.mark.parametrize("copies", [1500, 8000])
def test_many_ties_exact(dl, orc, metric, copies):
    g = W.rng(9400 + copies)
    X = W.dirichlet_histograms(g, 300, 8)
    check(dl, orc, X[:30], np.concatenate([X, np.repeat(X[:1], copies, axis=0)]), 10, metric)


def test_more_ties_than_the_list_holds_is_refused(dl):
    X = W.dirichlet_histograms(W.rng(9500), 20, 8)
    S = np.concatenate([X, np.repeat(X[:1], 9000, axis=0)])
    Q, Ss = _store(dl, np.arange(20), X), _store(dl, np.arange(len(S)), S)
    with pytest.raises(dl.DLError) as ei:
        dl.topk_join(Q, Ss, 3, metric="l1")
    assert ei.value.status == dl.DL_EOVERFLOW
