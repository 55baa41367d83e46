"""The autotuner's classes: FP16 and BF16 are timed apart, and an old cache file decides nothing.

A cache line of the first key format names a configuration that was timed with kernels since replaced.
"""

import ast
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TRIALS = [(256, 8), (128, 8), (256, 16), (256, 8)]   # top-k: every candidate once, then the first again

CODE = """
import torch
from paper_1812_07607_gb300 import dl, build
build.build()
g = torch.Generator(device="cuda"); g.manual_seed(1)
S = dl.Store(torch.arange(5000, device="cuda"), torch.rand(5000, 64, generator=g, device="cuda"))
Q = dl.Store(torch.arange(300, device="cuda"), torch.rand(300, 64, generator=g, device="cuda"))
out = {}
for p in ("fp16", "bf16"):
    out[p] = []
    for _ in range(6):
        r = dl.topk_join(Q, S, 4, precision=p)
        out[p].append((r.stats()["tile_n"], r.stats()["epilogue_warps"]))
        r.free()
print(torch.cuda.get_device_properties(0).multi_processor_count)
print(out)
"""


def run(cache):
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, env=dict(os.environ, DL_TUNE_CACHE=str(cache)), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    sms, out = r.stdout.strip().splitlines()[-2:]
    return int(sms), ast.literal_eval(out)


def test_formats_apart_and_old_lines_ignored(tmp_path):
    cache = tmp_path / "tune.txt"
    sms, out = run(cache)
    for p in ("fp16", "bf16"):
        assert out[p][:4] == TRIALS and out[p][4] == out[p][5] and out[p][4] in TRIALS, out
    lines = [ln.split() for ln in cache.read_text().splitlines()]
    assert len(lines) == 2 and len({k for k, _ in lines}) == 2
    cache.write_text(f"sm{sms}:dp64:k2:r8:s12 128\n")   # 300 rows against 5,000 x 64, as a file of before has it
    assert run(cache)[1]["fp16"][:4] == TRIALS
    again = run(cache)[1]   # the lines that the run before appended count
    assert len(set(again["fp16"])) == 1 and len(set(again["bf16"])) == 1
