"""The inner-product join runs on the 16-bit copy that the stores hold: no second one is built for it.

Kernels are counted (past 1,024 rows): the first call derives the column store's column arrays (one kernel more than a
later call) and nothing else. The sets equal the oracle's in either format, and where the two stores
hold different formats; explicit FP16 and d > 512 stay refused.
"""

import numpy as np
import pytest

import oracle
from paper_1812_07607_gb300 import workloads as W
from test_gpu_ip import _gpu, _rows, _store, _want, dl, orc  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


def launches(dl, R, S, t):
    n = dl.kernel_launches()
    res = dl.sim_join(R, S, t, metric="ip")
    prec = res.stats()["precision"]
    res.free()
    return dl.kernel_launches() - n, prec


@pytest.mark.parametrize("self_join", [False, True])
def test_first_call_builds_no_copy(dl, self_join):
    g = W.rng(9700)
    R, S = _store(dl, np.arange(300), _rows(g, 300, 64)), _store(dl, np.arange(1025), _rows(g, 1025, 64))
    first, prec = launches(dl, S if self_join else R, None if self_join else S, 1e9)
    later, _ = launches(dl, S if self_join else R, None if self_join else S, 1e9)
    assert first == later + 1 and prec == dl.DL_PREC_FP16


@pytest.mark.parametrize("d", [16, 130, 512])
def test_formats_exact(dl, orc, d):
    g = W.rng(9710 + d)
    R, S = _rows(g, 257, d), _rows(g, 2049, d)
    wide = R.copy()
    wide[5] *= np.float32(2.0 ** -40)   # past FP16's range: this store holds BF16
    rid, sid = np.arange(257, dtype=np.int64), np.arange(2049, dtype=np.int64) + 1000
    for Q, kw, want_prec in ((R, {}, dl.DL_PREC_FP16), (R, {"precision": "bf16"}, dl.DL_PREC_BF16), (wide, {}, dl.DL_PREC_BF16)):
        t = float(np.quantile(Q.astype(np.float64) @ S.astype(np.float64).T, 0.99))
        got, st = _gpu(dl, Q, S, t, rid, sid, **kw)
        assert got == _want(orc, Q, S, t, oracle.MODE_RXS, rid, sid) and st["precision"] == want_prec
    for A, kw in ((R, {"precision": "fp16"}), (_rows(g, 20, 640), {})):
        with pytest.raises(dl.DLError) as ei:
            dl.sim_join(_store(dl, np.arange(len(A)), A), None, 0.5, metric="ip", **kw)
        assert ei.value.status == dl.DL_EUNSUPPORTED
