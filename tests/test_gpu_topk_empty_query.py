"""Calls without query rows leave nothing behind: they succeed, and so do the calls after them.

A CUDA error that a call ignores stays with the thread and surfaces in the next call's launches.
"""

import numpy as np
import pytest

from paper_1812_07607_gb300 import workloads as W
from test_gpu_topk import _store, check_topk, dl, orc  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [{}, {"timing": True}, {"precision": "fp32", "timing": True}, {"tile_n": 128},
                                {"metric": "l1"}])
@pytest.mark.parametrize("nS", [0, 700])
def test_topk_without_query_rows(dl, orc, kw, nS):
    X = W.dirichlet_histograms(W.rng(8500), 700, 24)
    S, Q = _store(dl, np.arange(nS), X[:nS]), _store(dl, np.arange(0), X[:0])
    for _ in range(6):   # every trial of the tuner
        res = dl.topk_join(Q, S, 3, **kw)
        ids, d2 = res.topk_host()
        st = res.stats()
        res.free()
        assert ids.shape == d2.shape == (0, 3) and st["pairs_evaluated"] == 0
    check_topk(dl, orc, X[:5], X, 3)
    res = dl.sim_join(_store(dl, np.arange(700), X), None, 0.0)
    res.free()


@pytest.mark.parametrize("timing", [False, True])
def test_batch_and_join_without_query_rows(dl, orc, timing):
    X = W.dirichlet_histograms(W.rng(8501), 700, 24)
    S = _store(dl, np.arange(700), X)
    for kind in ("topk", "eps"):
        res = dl.batch_join(S, np.arange(4), X[:4], [{"kind": kind, "q_begin": 0, "nq": 0, "k": 3, "eps": 0.1}], timing=timing)
        res.free()
    res = dl.sim_join(_store(dl, np.arange(0), X[:0]), S, 0.1, timing=timing)
    res.free()
    check_topk(dl, orc, X[:5], X, 3)
