"""16-bit formats inside a batch: one request's rows decide neither another's answer nor refuse it."""

import numpy as np
import pytest

from paper_1812_07607_gb300 import workloads as W
from test_gpu_topk import _store, dl, orc  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


def data():
    g = W.rng(9800)
    S = W.dirichlet_histograms(g, 3000, 40)
    near, wide = W.dirichlet_histograms(g, 30, 40), W.dirichlet_histograms(g, 30, 40)
    wide[4] *= np.float32(2.0 ** -30)   # past FP16's range beside the other rows
    return S, near, wide


def test_fp16_server_answers_wide_rows_beside_others(dl, orc):
    S, near, wide = data()
    sv = dl.Server(_store(dl, np.arange(3000), S), slots=1, precision="fp16")
    tickets = [(sv.submit(np.arange(30), Q, "topk", k=5), Q) for Q in (near, wide, near)]
    for t, Q in tickets:
        res = None
        for _ in range(300):
            res = sv.poll(t, timeout_us=100_000)
            if res is not None:
                break
        ids, d2 = res.topk_host()
        oi, od = orc.topk(Q, S, 5)
        assert (ids == oi).all() and (d2 == od).all()
        res.free()
    sv.close()


@pytest.mark.parametrize("rows,want", [("near", "DL_PREC_FP16"), ("wide", "DL_PREC_BF16")])
@pytest.mark.parametrize("kinds", [("topk",), ("eps",), ("eps", "topk")])
def test_reported_precision(dl, rows, want, kinds):
    S, near, wide = data()
    Q = near if rows == "near" else wide
    res = dl.batch_join(_store(dl, np.arange(3000), S), np.arange(30), Q,
                        [{"kind": kind, "q_begin": 0, "nq": 30, "k": 4, "eps": 0.1} for kind in kinds])
    assert res.stats()["precision"] == getattr(dl, want)
    res.free()
