"""The histogram top-k takes fewer query rows at a time where memory is short.

Its scratch of distances and lists is 330 MB where there are rows for it; with 200 MB left a call has
to give the same answer. In a process of its own: the pool keeps what earlier calls took.
"""

import os
import subprocess
import sys

import pytest

from test_gpu_topk import dl  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("metric", ["l1", "chi2"])
def test_short_memory(dl, metric):
    same, = subprocess.run([sys.executable, "-c", f"""
import torch
from paper_1812_07607_gb300 import dl
g = torch.Generator(device="cuda"); g.manual_seed(8)
X = torch.rand(70000, 16, generator=g, device="cuda")
st = lambda x: dl.Store(torch.arange(len(x), device="cuda"), x)
Q, S, few = st(X[:1500].contiguous()), st(X), st(X[:40].contiguous())
def call(Q):
    r = dl.topk_join(Q, S, 10, metric="{metric}"); a = r.topk_host(); r.free(); return a
want = call(few)
hold = torch.empty(torch.cuda.mem_get_info()[0] - (200 << 20), dtype=torch.uint8, device="cuda")
ids, d2 = call(Q)
print(bool((ids[:40] == want[0]).all() and (d2[:40] == want[1]).all() and (ids >= 0).all()))
"""], cwd=ROOT, capture_output=True, text=True, timeout=600, check=True).stdout.split()
    assert same == "True"
