"""The epsilon epilogue's rows put aside, and the passes behind it, exact against the oracle.

A 32 x 32 chunk of a tile puts up to four hit rows aside and classifies them after the accumulator is
released; more go through the many-row path. Cluster counts from one (every pair matches) to none take
a chunk through every number of hit rows, with eight and sixteen epilogue warps. The full mode (two
pairs a match) and a buffer too small for the pairs run over clustered rows too. A 70,000-row clustered store has R tiles whose first columns lie past a block of
tile tests, and features that start off a 16-byte line take the unaligned reads.
"""

import numpy as np
import pytest

from paper_1812_07607_gb300 import workloads as W
from test_gpu_topk import _store, check_topk, dl, orc  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


def _clustered(g, n, d, clusters):
    C = g.standard_normal((clusters, d))
    X = C[g.integers(0, clusters, n)] + 1e-3 * g.standard_normal((n, d))
    return (X / np.linalg.norm(X, axis=1, keepdims=True)).astype(np.float32)


def _got(res):
    a, b = res.pairs_host()
    res.free()
    return np.sort(a.astype(np.int64) * 2**32 + b)


@pytest.mark.parametrize("warps", [8, 16])
@pytest.mark.parametrize("clusters", [1, 3, 40, 170, 340, 1000, 4000])
@pytest.mark.parametrize("n,m,d", [(700, 900, 64), (333, 1025, 200)])
def test_hit_rows_exact(dl, orc, n, m, d, clusters, warps):
    g = W.rng(9300 + clusters + d)
    X = _clustered(g, n + m, d, clusters)
    R, S = X[:n], X[n:]
    D = orc.dist_block(R, S)
    eps = 0.1   # rows of a cluster lie within 0.1 (d x 2e-6 squared), others farther or as the oracle says
    want = np.argwhere(D <= np.float64(eps * eps))
    want = np.sort(want[:, 0] * 2**32 + want[:, 1])
    Rs, Ss = _store(dl, np.arange(n), R), _store(dl, np.arange(m), S)
    assert np.array_equal(_got(dl.sim_join(Rs, Ss, eps, tile_n=256, epilogue_warps=warps)), want)


@pytest.mark.parametrize("clusters", [2, 300])
def test_full_mode_and_small_buffer(dl, orc, clusters):
    n = 600
    X = _clustered(W.rng(9400 + clusters), n, 48, clusters)
    want = np.argwhere(orc.dist_block(X, X) <= np.float64(0.1 * 0.1))
    want = np.sort(want[:, 0] * 2**32 + want[:, 1])
    S = _store(dl, np.arange(n), X)
    assert np.array_equal(_got(dl.sim_join(S, None, 0.1, self_mode="full")), want)
    for cap in (1, 127, 333):
        res = dl.sim_join(S, None, 0.1, self_mode="full", out_capacity=cap, allow_overflow=True)
        assert res.count() == len(want)
        a, b = res.pairs_host()
        res.free()
        part = a.astype(np.int64) * 2**32 + b
        assert len(part) == min(cap, len(want)) and len(np.unique(part)) == len(part) and np.isin(part, want).all()


def test_pruned_self_join_past_a_block_of_tiles(dl):
    X = _clustered(W.rng(9500), 70_000, 16, 500)
    S = _store(dl, np.arange(70_000), X).clustered(500, iters=2)
    res = dl.sim_join(S, None, 0.01, prune=True)
    pruned = _got(res)
    assert len(pruned) > 1000 and np.array_equal(pruned, _got(dl.sim_join(S, None, 0.01)))


@pytest.mark.parametrize("d", [1, 31, 64, 127, 130])
@pytest.mark.parametrize("off", [1, 2, 3])
def test_features_off_a_line(dl, orc, d, off):
    import torch
    n = 301
    X = _clustered(W.rng(9600 + d), n, d, 60)
    flat = torch.zeros(n * d + off, device="cuda")
    flat[off:] = torch.from_numpy(X).cuda().reshape(-1)
    S = dl.Store(torch.arange(n).cuda(), flat[off:].view(n, d))
    a, b = np.nonzero(np.triu(orc.dist_block(X, X) <= np.float64(0.1 * 0.1), 1))
    assert np.array_equal(_got(dl.sim_join(S, None, 0.1)), np.sort(a * 2**32 + b))


@pytest.mark.parametrize("kind", ["spread", "gaps", "tiny"])
def test_topk_terms_over_the_exponents(dl, orc, kind):
    g = W.rng(9700)
    nQ, nS, d = 40, 3000, 36
    X = g.standard_normal((nQ + nS, d))
    if kind == "spread":     # exponents up to 60 apart: both sides of the integer terms' limit
        X *= np.exp2(g.integers(-30, 31, X.shape))
    elif kind == "gaps":     # exact zeros, and neighbours that cancel
        X[g.random(X.shape) < 0.4] = 0.0
        X[nQ:nQ + 500] = np.nextafter(X[g.integers(0, nQ, 500)].astype(np.float32), np.float32(9))
    else:                    # subnormal features
        X *= 2.0 ** -130
    X = X.astype(np.float32)
    check_topk(dl, orc, X[:nQ], X[nQ:], 25)
