"""The FP16 tensor-core path: its error bound, its scales and its fallback to BF16, all exact.

AUTO takes FP16 copies (x = s x16, one power of two s per store) where a store's rows lie within
2^18 of each other in their largest magnitudes, else BF16. The bound is checked as in
test_gpu_bounds.py: |h~ - h| <= E for 1.05e8 pairs a case, and the accumulation error alone stays
below 5% of the assumed d_p 2^-20 ||q~|| ||x~||. The joins are compared with the oracle at ragged
sizes, around the range line, at both ends of the feature domain, and between stores of different
formats.
"""

import numpy as np
import pytest

import oracle
from paper_1812_07607_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dl():
    import torch
    from paper_1812_07607_gb300 import build as B, dl as D
    assert torch.cuda.is_available()
    B.build()
    D.load()
    return D


@pytest.fixture(scope="module")
def orc():
    return oracle.default()


def _store(dl, X, base=0):
    import torch
    return dl.Store(torch.arange(len(X)).cuda() + base, torch.from_numpy(np.ascontiguousarray(X)).cuda())


def enc(X):
    """Host rebuild of the FP16 copy: s = 2^(e - 15) with the store's largest magnitude in [2^(e-1), 2^e);
    for 256 < d <= 512 the codes keep 9 significant bits (magnitudes rounded half up)."""
    s = np.ldexp(1.0, int(np.frexp(np.abs(X).max())[1]) - 15)
    y = (X.astype(np.float64) / s).astype(np.float32)
    sh = 24 - (9 if 256 < X.shape[1] <= 512 else 11)
    y = (((y.view(np.uint32) + np.uint32(1 << (sh - 1))) >> np.uint32(sh)) << np.uint32(sh)).view(np.float32)
    return y.astype(np.float16).astype(np.float64) * s


@pytest.mark.parametrize("d", [64, 128, 256, 512, 1024])
@pytest.mark.parametrize("kind", ["hist", "signed"])
def test_bound_and_accumulation_margin(dl, d, kind):
    import torch
    g = W.rng(9100 + d + (kind == "signed"))
    n = 10240
    R, S = ((W.dirichlet_histograms(g, n, d) for _ in range(2)) if kind == "hist"
            else (W.unit_mixture(g, n, d, 64, 0.05)[0] for _ in range(2)))
    h, e = dl.debug_scores(_store(dl, R), _store(dl, S), "fp16")
    h, e = h.double(), e.double()
    R64, S64 = torch.from_numpy(R).cuda().double(), torch.from_numpy(S).cuda().double()
    beta = 0.5 * (S64 * S64).sum(dim=1)
    ratio = float(((h - (R64 @ S64.T - beta[None, :])).abs() / e).max())
    Rq, Sq = torch.from_numpy(enc(R)).cuda(), torch.from_numpy(enc(S)).cuda()
    acc = (h - (Rq @ Sq.T - beta.float().double()[None, :])).abs()
    gamma = (d + 63) // 64 * 64 * 2.0 ** -20
    acc_ratio = float((acc / (gamma * Rq.norm(dim=1)[:, None] * Sq.norm(dim=1)[None, :])).max())
    print(f"fp16 d={d} {kind}: max |h~-h|/E {ratio:.3f}; max accumulation / assumed {acc_ratio:.2e}")
    assert ratio <= 1.0
    assert acc_ratio < 0.05


def check(dl, orc, R, S, q, precision="auto", want_prec=None):
    D = orc.dist_block(R, S)
    eps = float(np.sqrt(np.quantile(D, q)))
    res = dl.sim_join(_store(dl, R), _store(dl, S, 10**6), eps, precision=precision)
    a, b = res.pairs_host()
    st = res.stats()
    res.free()
    p = orc.join(R, S, eps)
    assert len(a) == len(p) and set(zip(a.tolist(), (b - 10**6).tolist())) == set(map(tuple, p.tolist())), st
    if want_prec is not None:
        assert st["precision"] == want_prec
    return st


@pytest.mark.parametrize("n,m,d", [(1, 1, 1), (33, 257, 5), (129, 130, 63), (300, 700, 65), (255, 1000, 200), (127, 511, 512)])
def test_ragged_exact(dl, orc, n, m, d):
    g = W.rng(9200 + n + m + d)
    check(dl, orc, W.dirichlet_histograms(g, n, d), W.dirichlet_histograms(g, m, d), 0.01, want_prec=dl.DL_PREC_FP16)


@pytest.mark.parametrize("d", [513, 768, 1024])
def test_streamed_above_512_exact(dl, orc, d):
    g = W.rng(9250 + d)
    R, c = W.unit_mixture(g, 300, d, 16, 0.1 / np.sqrt(d))
    S, _ = W.unit_mixture(g, 900, d, 16, 0.1 / np.sqrt(d), centroids=c)
    check(dl, orc, R, S, 0.02, precision="fp16", want_prec=dl.DL_PREC_FP16)


def test_auto_takes_fp16_above_512_for_large_joins(dl):
    import torch
    g = W.rng(9260)
    X, _ = W.unit_mixture(g, 9000, 600, 64, 0.1 / np.sqrt(600))
    Xs = _store(dl, X)
    sets = {}
    for p in ("auto", "fp8", "fp32"):
        res = dl.sim_join(Xs, Xs, 0.14, precision=p)
        a, b = res.pairs_device()
        sets[p] = torch.sort(a * 9000 + b).values.cpu()
        if p == "auto":
            assert res.stats()["precision"] == dl.DL_PREC_FP16
        del a, b, res
    assert len(sets["auto"]) > 9000 and torch.equal(sets["auto"], sets["fp32"]) and torch.equal(sets["fp8"], sets["fp32"])


@pytest.mark.parametrize("mag", [2.0 ** -60, 2.0 ** -46, 2.0 ** -20, 1.0, 2.0 ** 20, 2.0 ** 39])
def test_any_scale_exact(dl, orc, mag):
    g = W.rng(9270)
    X = (W.dirichlet_histograms(g, 700, 96) * np.float32(mag)).astype(np.float32)
    # 2^-46: the largest features sit on either side of the 2^-47 line
    want = None if mag == 2.0 ** -46 else dl.DL_PREC_BF16 if mag < 2.0 ** -50 else dl.DL_PREC_FP16
    check(dl, orc, X[:200], X[200:], 0.01, want_prec=want)


@pytest.mark.parametrize("span,f16", [(16, True), (24, False)])
def test_wide_ranges_exact(dl, orc, span, f16):
    """Rows whose magnitudes span 2^16 (FP16) and 2^24 (BF16), zero rows among them."""
    g = W.rng(9280)
    X = W.dirichlet_histograms(g, 900, 40)
    X = (X / X.max(axis=1, keepdims=True) * np.exp2(-np.linspace(0, span, 900))[:, None]).astype(np.float32)
    X[::50] = 0
    X = X[g.permutation(900)]
    check(dl, orc, X[:300], X[300:], 0.3, want_prec=dl.DL_PREC_FP16 if f16 else dl.DL_PREC_BF16)
    if not f16:
        with pytest.raises(dl.DLError) as ei:
            dl.sim_join(_store(dl, X), None, 0.1, precision="fp16")
        assert ei.value.status == dl.DL_EUNSUPPORTED


def test_stores_of_different_formats_exact(dl, orc):
    """One store holds FP16, the other BF16: the join, a top-k and a batch run in BF16."""
    import torch
    g = W.rng(9290)
    R = W.dirichlet_histograms(g, 300, 48)
    S = W.dirichlet_histograms(g, 900, 48)
    S[:40] *= np.float32(2.0 ** -25)
    check(dl, orc, R, S, 0.02, want_prec=dl.DL_PREC_BF16)
    res = dl.topk_join(_store(dl, R), _store(dl, S), 7)
    ids, d2 = res.topk_host()
    res.free()
    oi, od = orc.topk(R, S, 7)
    assert (ids == oi).all() and (d2 == od).all()
    eps = 0.2
    br = dl.batch_join(_store(dl, S), torch.arange(300).cuda(), torch.from_numpy(R).cuda(),
                       [{"kind": "eps", "q_begin": 0, "nq": 300, "eps": eps}])
    a, b = br.request_pairs(0)
    assert set(zip(a.tolist(), b.tolist())) == set(map(tuple, orc.join(R, S, eps).tolist()))


def test_batch_rows_shared_by_requests_exact(dl, orc):
    """Requests that share rows: more query rows than the call brings."""
    import torch
    g = W.rng(9295)
    Q, S = W.dirichlet_histograms(g, 150, 32), W.dirichlet_histograms(g, 800, 32)
    reqs = [{"kind": "eps", "q_begin": 10 * i, "nq": 150 - 10 * i, "eps": 0.1 + 0.02 * i} for i in range(5)]
    br = dl.batch_join(_store(dl, S), torch.arange(150).cuda(), torch.from_numpy(Q).cuda(), reqs)
    for i, r in enumerate(reqs):
        a, b = br.request_pairs(i)
        p = orc.join(Q[r["q_begin"]:], S, r["eps"])
        assert set(zip((a - r["q_begin"]).tolist(), b.tolist())) == set(map(tuple, p.tolist()))
