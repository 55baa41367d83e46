"""The two-pass top-k at its edges, ids and FP64 distances bit-exact against the oracle.

Stores that fit a row's list whole (no first pass) and just do not; group maxima of 16 and of 64
columns; strides above one; k from 1 to 1024 with fewer groups than k; rows whose list overflows
because near-duplicates lie side by side (a store in cluster order), which take tightened thresholds;
exact duplicates past every list, which take the exact scan; BF16 operands; and more query rows than
a chunk of the workspace holds.
"""

import numpy as np
import pytest

from paper_1812_07607_gb300 import workloads as W
from test_gpu_topk import _store, check_topk, dl, orc  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nQ,nS,d,k", [
    (5, 160, 16, 1), (5, 161, 16, 1), (129, 192, 8, 10), (129, 193, 8, 10),    # around a list's capacity
    (1, 4096, 64, 1), (3, 20_000, 128, 1), (130, 66_000, 130, 2),              # strides 1 to 16
    (7, 2300, 33, 1024), (4, 30_000, 20, 1024), (2, 40_000, 512, 100), (17, 9000, 300, 37),
])
@pytest.mark.parametrize("precision", ["auto", "bf16"])
def test_shapes_exact(dl, orc, nQ, nS, d, k, precision):
    g = W.rng(8100 + nQ + nS + d + k)
    X, _ = W.clustered_histograms(g, nQ + nS, d, max(2, nS // 40), 0.01)
    check_topk(dl, orc, X[:nQ], X[nQ:], k, precision=precision)


@pytest.mark.parametrize("k", [3, 100])
def test_cluster_order_overflows_then_refines(dl, orc, k):
    g = W.rng(8200 + k)
    X, _ = W.clustered_histograms(g, 20_000, 24, 66, 0.002)
    Q = X[:150] * np.float32(1.0001)
    sid = np.arange(20_000) * 7 + 5
    S = _store(dl, sid, X).clustered(128, iters=2)
    res = dl.topk_join(_store(dl, np.arange(150), Q), S, k)
    ids, d2 = res.topk_host()
    res.free()
    oi, od = orc.topk(Q, X, k)
    assert (ids == sid[oi]).all() and (d2 == od).all()


def test_duplicates_past_every_list_exact(dl, orc):
    g = W.rng(8300)
    B = W.dirichlet_histograms(g, 30, 12)
    S = np.concatenate([np.repeat(B[:3], 2500, axis=0), W.dirichlet_histograms(g, 9000, 12)])
    st = check_topk(dl, orc, B, S, 20)
    assert 3 <= st["band_pairs"] < 30


def test_more_rows_than_a_chunk_exact(dl, orc):
    import torch
    g = W.rng(8400)
    S = W.dirichlet_histograms(g, 2400, 6)
    Q = W.dirichlet_histograms(g, 40_000, 6)
    res = dl.topk_join(_store(dl, np.arange(40_000), Q), _store(dl, np.arange(2400), S), 1024)
    ids, d2 = res.topk_host()
    res.free()
    rows = np.concatenate([np.arange(20), g.choice(40_000, 60, replace=False), np.arange(39_980, 40_000)])
    oi, od = orc.topk(Q[rows], S, 1024)
    assert (ids[rows] == oi).all() and (d2[rows] == od).all()
