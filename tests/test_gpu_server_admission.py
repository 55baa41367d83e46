"""What the server admits: a top-k request is refused for its workspace by the line it always was.

The estimate of the two-pass lists is larger at small k than that of the heaps before them, but the
lists are cut to the memory there is: a request that fitted the budget then is admitted and answered.
"""

import numpy as np
import pytest

from paper_1812_07607_gb300 import workloads as W
from test_gpu_topk import _store, dl, orc  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


def test_topk_requests_within_the_heaps_estimate_are_admitted(dl, orc):
    g = W.rng(8700)
    S, Q = W.dirichlet_histograms(g, 300_000, 16), W.dirichlet_histograms(g, 7000, 16)
    sv = dl.Server(_store(dl, np.arange(300_000), S), mem_budget_bytes=64 << 20, slots=1, max_batch_rows=20_000)
    t = sv.submit(np.arange(7000), Q, "topk", k=1)   # 16 x (4 + 512) bytes of heaps and lists a row, 3.7 MB of rows and output: 61.5 MB
    res = None
    for _ in range(600):
        res = sv.poll(t, timeout_us=100_000)
        if res is not None:
            break
    ids, d2 = res.topk_host()
    rows = g.choice(7000, 40, replace=False)
    oi, od = orc.topk(Q[rows], S, 1)
    assert (ids[rows] == oi).all() and (d2[rows] == od).all()
    res.free()
    with pytest.raises(dl.DLError) as ei:   # 16 x (40 + 512) bytes a row, in either estimate more than the budget
        sv.submit(np.arange(9000), np.concatenate([Q, Q[:2000]]), "topk", k=10)
    assert ei.value.status == dl.DL_ENOMEM_ADMIT
    sv.close()
