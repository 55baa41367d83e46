"""The top-k's workspace is bounded whatever the data, and follows what the device has left.

Where the 16-bit bound exceeds the spread of the distances (rows with a large common offset), a row's
threshold admits every column. The candidates then have to stay within the workspace's limit, the
rows concerned take the exact scan, the others their lists, and ids and distances stay bit-exact.
Memory is looked at from processes of their own: the pool keeps what earlier calls took.
"""

import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1812_07607_gb300 import workloads as W
from test_gpu_topk import _store, check_topk, dl, orc  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(code):
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout.split()


def offset(g, n, d):
    return (1000 + 1e-3 * g.standard_normal((n, d))).astype(np.float32)


def test_offset_cluster_memory_is_bounded(dl):
    """1,536 rows that each reach all of 200,000 columns: 2.5 GB as one list of 8-byte candidates."""
    taken, = run("""
import torch
from paper_1812_07607_gb300 import dl
g = torch.Generator(device="cuda"); g.manual_seed(5)
st = lambda n: dl.Store(torch.arange(n, device="cuda"), 1000 + torch.randn(n, 16, generator=g, device="cuda") * 1e-3)
Q, S = st(1536), st(200000)
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
dl.topk_join(Q, S, 10).free()
print(free - torch.cuda.mem_get_info()[0])
""")
    # the lists' limit (2^30) and the exact scan's (2^28), in the pool's granularity
    assert int(taken) <= (1 << 30) + (1 << 28) + (1 << 27)


@pytest.mark.parametrize("k", [1, 40])
@pytest.mark.parametrize("bad", [3, 150, 300])
def test_rows_past_the_shared_list_exact(dl, orc, bad, k):
    g = W.rng(8600 + bad + k)
    S = np.concatenate([offset(g, 20_000, 16), W.dirichlet_histograms(g, 9000, 16)])
    Q = np.concatenate([offset(g, bad, 16), W.dirichlet_histograms(g, 300 - bad, 16)])
    st = check_topk(dl, orc, Q, S, k)
    assert st["band_pairs"] <= bad


def test_rows_that_no_threshold_helps_are_scanned_at_once(dl, orc):
    """Every row reaches every column: a first listing, one with the list's size, no tightened ones."""
    g = W.rng(8630)
    S, Q = offset(g, 20_000, 16), offset(g, 300, 16)
    st = check_topk(dl, orc, Q, S, 10)
    assert st["band_pairs"] == 300 and st["kernels_launched"] <= 1 + 7 + 7 + 1   # setup, passes, the scan


def test_no_lists_where_every_column_passes(dl, orc):
    """Known after the first listing: no second one, and rows with near columns are still exact."""
    g = W.rng(8635)
    S = np.concatenate([offset(g, 20_000, 16), W.dirichlet_histograms(g, 50, 16)])
    Q = np.concatenate([offset(g, 300, 16), W.dirichlet_histograms(g, 3, 16)])
    st = check_topk(dl, orc, Q, S, 10)
    assert st["band_pairs"] == 303 and st["kernels_launched"] <= 1 + 7 + 1 + 1   # setup, passes, the names, the scan


def test_more_columns_than_the_list_ever_holds(dl, orc):
    """One tile of rows that reach 1.2 million columns each: more than a gigabyte of candidates."""
    g = W.rng(8640)
    S = np.concatenate([offset(g, 1_200_000, 8), W.dirichlet_histograms(g, 1000, 8)])
    Q = np.concatenate([offset(g, 126, 8), W.dirichlet_histograms(g, 4, 8)])
    res = dl.topk_join(_store(dl, np.arange(130), Q), _store(dl, np.arange(len(S)), S), 3)
    ids, d2 = res.topk_host()
    res.free()
    rows = [0, 1, 60, 125, 126, 129]
    oi, od = orc.topk(Q[rows], S, 3)
    assert (ids[rows] == oi).all() and (d2[rows] == od).all()


def test_all_rows_past_the_shared_list_in_a_batch(dl, orc):
    g = W.rng(8650)
    S, Q = offset(g, 15_000, 24), offset(g, 260, 24)
    res = dl.batch_join(_store(dl, np.arange(15_000), S), np.arange(260), Q,
                        [{"kind": "topk", "q_begin": 0, "nq": 130, "k": 7}, {"kind": "topk", "q_begin": 130, "nq": 130, "k": 100}])
    for i, k in ((0, 7), (1, 100)):
        ids, d2 = res.request_topk(i)
        oi, od = orc.topk(Q[130 * i:130 * i + 130], S, k)
        assert (ids == oi).all() and (d2 == od).all()
    res.free()


def test_short_memory_takes_fewer_rows_at_a_time(dl):
    """A call whose lists would take a gigabyte, on a device with a third of one left."""
    same, = run("""
import torch
from paper_1812_07607_gb300 import dl
g = torch.Generator(device="cuda"); g.manual_seed(6)
X = torch.rand(60000, 16, generator=g, device="cuda")
st = lambda x: dl.Store(torch.arange(len(x), device="cuda"), x)
Q, S = st(X[:16000].contiguous()), st(X)
def call(Q):
    r = dl.topk_join(Q, S, 512); a = r.topk_host(); r.free(); return a
small = call(st(X[:200].contiguous()))          # modules loaded, little in the pool
free = torch.cuda.mem_get_info()[0]
out = 16000 * 512 * 16
hold = torch.empty(free - out - (340 << 20), dtype=torch.uint8, device="cuda")
ids, d2 = call(Q)
print(bool((ids[:200] == small[0]).all() and (d2[:200] == small[1]).all() and (ids >= 0).all()))
""")
    assert same == "True"
