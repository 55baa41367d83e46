"""The calls whose speed this framework is judged by, from one image query to full-size joins.

A case is a dict of plain values. `prepare` draws a case's inputs on the GPU from a seed (patch
features as in `workloads.py`: Dirichlet(0.5) colour histograms, jittered views of repeated
objects, unit-norm embedding mixtures) and builds the stores a program keeps; `run` makes one
call through the public API and returns everything the call computes. A join's result is a set,
in no fixed order, and a program that goes on with it puts it in one: `run` marks the pairs of a
small join in its match matrix, and returns those of a larger one sorted, each packed as
(row of R) << 32 | (row of S) with ids = row numbers, in a table of fixed size (-1 past the last).
"""

import ctypes
import math

import numpy as np
import torch

from paper_1812_07607_gb300 import dl, workloads as W

DEV = "cuda"
VIEWS = 32   # views (rows) of each object in the clustered stores, as in the 262,144-row workload
MATRIX = 1 << 24   # joins of at most this many pairs return their match matrix


def listed():
    return [
        # two small patch collections: a call that is all launches and latency (2,000 x 2,000, d = 64)
        {"name": "join_2k", "op": "join", "n": 2000, "m": 2000, "d": 64, "data": "plain", "metric": "l2", "per_row": 2},
        # near-duplicates within one collection (q4): the 262,144 x 128 self-join, 20 matches a patch
        {"name": "self_262k", "op": "join", "n": 262144, "m": 0, "d": 128, "data": "objects", "metric": "l2", "per_row": 20},
        # embeddings of two videos compared by cosine similarity, ragged sizes, d = 512
        {"name": "cosine_d512", "op": "join", "n": 131072, "m": 200003, "d": 512, "data": "unit", "metric": "cosine", "per_row": 10},
        # wide embeddings (the FP8 tensor-core path, which d > 512 takes by default)
        {"name": "join_d1024", "op": "join", "n": 65536, "m": 50001, "d": 1024, "data": "unit", "metric": "l2", "per_row": 10},
        # colour histograms compared by their L1 distance, which has no tensor-core form
        {"name": "l1_self_64k", "op": "join", "n": 65536, "m": 0, "d": 128, "data": "objects", "metric": "l1", "per_row": 20},
        # the index join: many views of few tracked objects, store in cluster order
        {"name": "pruned_131k", "op": "pruned", "n": 131072, "d": 128, "per_row": 100},
        # reverse image search (q1): the closest of a million patches to one query image
        {"name": "search_1m", "op": "topk", "n": 1, "m": 1000003, "d": 256, "k": 1, "metric": "l2"},
        # a stack of queries, each with its 100 nearest patches of a million
        {"name": "topk_4096", "op": "topk", "n": 4096, "m": 1000003, "d": 256, "k": 100, "metric": "l2"},
        # image search under the chi-square histogram distance
        {"name": "chi2_top10", "op": "topk", "n": 1000, "m": 65536, "d": 128, "k": 10, "metric": "chi2"},
        # a batch of requests of uneven sizes against one store: epsilon-joins at 0.05 to 0.5 %
        # selectivity and top-10 searches
        {"name": "batch_64", "op": "batch", "requests": 64, "mix": 7, "m": 262144, "d": 128},
        # colour histograms of detector boxes on 1080p frames
        {"name": "color_hist", "op": "hist", "frames": 64, "boxes": 64, "h": 1080, "w": 1920, "bins": 8, "mix": 5},
        # q4 from features to objects: ingest, self-join, connected components
        {"name": "dedup_100k", "op": "dedup", "n": 100003, "d": 128, "per_row": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["join", "join", "self", "hist_join", "pruned", "topk", "topk", "hist_topk", "batch", "hist", "dedup"])
    if op == "join":
        data = rng.choice(["plain", "objects", "unit"])
        n, m, d = _log(rng, 500, 262144), _log(rng, 500, 262144), _log(rng, 16, 1024)
        while n * m * d > 131072 * 200003 * 512 or (data != "unit" and d > 512):
            n, m, d = _log(rng, 500, 262144), _log(rng, 500, 262144), _log(rng, 16, 1024)
        return {"op": "join", "n": n, "m": m, "d": d, "data": data, "metric": "cosine" if data == "unit" and rng.random() < 0.5 else "l2",
                "per_row": rng.randint(1, 20)}
    if op == "self":
        return {"op": "join", "n": _log(rng, 1000, 262144), "m": 0, "d": _log(rng, 16, 256), "data": "objects", "metric": "l2", "per_row": rng.randint(1, 20)}
    if op == "hist_join":
        return {"op": "join", "n": _log(rng, 1000, 65536), "m": 0, "d": _log(rng, 16, 128), "data": "objects", "metric": rng.choice(["l1", "chi2"]),
                "per_row": rng.randint(1, 20)}
    if op == "pruned":
        return {"op": "pruned", "n": _log(rng, 16384, 131072), "d": _log(rng, 32, 256), "per_row": rng.randint(10, 100)}
    if op == "topk":
        return {"op": "topk", "n": _log(rng, 1, 4096), "m": _log(rng, 10000, 1000003), "d": _log(rng, 32, 256), "k": rng.choice([1, 10, 100]), "metric": "l2"}
    if op == "hist_topk":
        return {"op": "topk", "n": _log(rng, 1, 1000), "m": _log(rng, 2000, 65536), "d": _log(rng, 16, 128), "k": rng.choice([1, 10, 100]),
                "metric": rng.choice(["l1", "chi2"])}
    if op == "batch":
        return {"op": "batch", "requests": _log(rng, 1, 64), "mix": rng.randrange(1000), "m": _log(rng, 20000, 262144), "d": _log(rng, 32, 128)}
    if op == "hist":
        h, w = rng.choice([(1080, 1920), (720, 1280), (481, 853)])
        return {"op": "hist", "frames": _log(rng, 1, 64), "boxes": rng.randint(8, 64), "h": h, "w": w, "bins": rng.choice([4, 6, 8]), "mix": rng.randrange(1000)}
    return {"op": "dedup", "n": _log(rng, 2000, 100003), "d": _log(rng, 16, 256), "per_row": rng.randint(1, 20)}


# ------------------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _centres(g, c, d):
    x = torch.randn(c, d, generator=g, device=DEV).square_()   # Gamma(1/2) draws: rows are Dirichlet(0.5)
    return x.div_(x.sum(1, keepdim=True))


def _views(g, cents, n, sigma):
    """n jittered views of the centres: N(0, sigma^2) per bin, clipped at 0, renormalised."""
    c, d = cents.shape
    pick = torch.randint(0, c, (n,), generator=g, device=DEV)
    x = torch.randn(n, d, generator=g, device=DEV).mul_(sigma).add_(cents[pick]).clamp_(min=0)
    return x.div_(x.sum(1, keepdim=True).clamp_(min=1e-6))


def _embeddings(g, cents, n):
    """n unit-norm rows of the mixture (jitter 0.02 per coordinate at d = 512, the same norm at any d)."""
    c, d = cents.shape
    pick = torch.randint(0, c, (n,), generator=g, device=DEV)
    x = torch.randn(n, d, generator=g, device=DEV).mul_(0.02 * math.sqrt(512 / d)).add_(cents[pick])
    return x.div_(x.norm(dim=1, keepdim=True))


def _rows(case, g):
    """(R, S or None) of a join case."""
    n, m, d = case["n"], case["m"], case["d"]
    if case["data"] == "plain":
        return _centres(g, n, d), (_centres(g, m, d) if m else None)
    if case["data"] == "unit":
        c = torch.randn(max(1, m // 256), d, generator=g, device=DEV)
        c.div_(c.norm(dim=1, keepdim=True))
        return _embeddings(g, c, n), (_embeddings(g, c, m) if m else None)
    c = _centres(g, max(1, max(n, m) // VIEWS), d)
    return _views(g, c, n, 0.01), (_views(g, c, m, 0.01) if m else None)


def _pair_dist(q, x, metric):
    """FP32 distances [len(q), len(x)] to set thresholds by (squared for l2 / cosine)."""
    if metric in ("l2", "cosine"):
        return ((q * q).sum(1)[:, None] + (x * x).sum(1)[None, :] - 2.0 * (q @ x.T)).clamp_(min=0)
    out = torch.empty(len(q), len(x), device=DEV)
    for i in range(len(q)):
        t = (q[i] - x).abs_()
        out[i] = t.sum(1) if metric == "l1" else (t * t / (q[i] + x).clamp_(min=1e-20)).sum(1)
    return out


def _threshold(R, S, metric, per_row):
    """The threshold that gives about per_row matches a row, from a sample of R's rows."""
    k = min(128 if metric in ("l2", "cosine") else 32, len(R))
    q = R[:k]
    x = R if S is None else S
    dist = _pair_dist(q, x, metric).flatten()
    want = min(len(dist) - 1, k * (per_row + (1 if S is None else 0)))   # a row's distance to itself is no match
    t = float(torch.topk(dist, want, largest=False).values[-1])
    t = {"l2": math.sqrt(t), "cosine": 1.0 - 0.5 * t}.get(metric, t)
    return float("%.6g" % t)


def _room(case):
    """Room for three times the matches that the threshold's sample promises."""
    return 4096 + 3 * case["n"] * case["per_row"]


def _store(x):
    return dl.Store(torch.arange(len(x), dtype=torch.int64, device=DEV), x)


def _mix(case):
    """Requests of a batch (sizes lognormal(5, 1.5) in [1, 8192], 70 % eps, 30 % top-10) and their rows."""
    reqs = W.request_mix(W.rng(case["mix"]), case["requests"], 5.0, 1.5, 8192, 0.3)
    return reqs, sum(r["nq"] for r in reqs)


def _boxes(case):
    return W.detector_boxes(W.rng(case["mix"]), case["frames"], case["h"], case["w"], case["boxes"])


def prepare(case, seed):
    g, op = _gen(seed), case["op"]
    if op == "join":
        R, S = _rows(case, g)
        eps = _threshold(R, S, case["metric"], case["per_row"])
        Rs, Ss = _store(R), (None if S is None else _store(S))
        if case["metric"] == "cosine":
            Rs, Ss = Rs.normalized(), (None if Ss is None else Ss.normalized())
        return {"op": op, "R": Rs, "S": Ss, "eps": eps, "metric": case["metric"], "room": _room(case)}
    if op == "pruned":
        X = _views(g, _centres(g, max(1, case["n"] // 1024), case["d"]), case["n"], 0.003)
        eps = _threshold(X, None, "l2", case["per_row"])
        return {"op": op, "X": _store(X).clustered(max(1, case["n"] // 256), iters=5), "eps": eps, "room": _room(case)}
    if op == "topk":
        c = _centres(g, max(1, case["m"] // VIEWS), case["d"])
        S, Q = _views(g, c, case["m"], 0.01), _views(g, c, case["n"], 0.01)
        return {"op": op, "Q": _store(Q), "S": _store(S), "k": case["k"], "metric": case["metric"]}
    if op == "batch":
        reqs, rows = _mix(case)
        c = _centres(g, max(1, case["m"] // VIEWS), case["d"])
        S, Q = _views(g, c, case["m"], 0.01), _views(g, c, rows, 0.01)
        dist = _pair_dist(Q[:32], S, "l2").flatten()
        kth = torch.topk(dist, int(5.1e-3 * len(dist)) + 1, largest=False).values
        table, at = [], 0
        for r in reqs:
            t = {"kind": r["kind"], "q_begin": at, "nq": r["nq"]}
            if r["kind"] == "topk":
                t["k"] = r["k"]
            else:
                t["eps"] = float("%.6g" % math.sqrt(float(kth[int(r["selectivity"] * len(dist))])))
            table.append(t)
            at += r["nq"]
        return {"op": op, "S": _store(S), "ids": torch.arange(rows, dtype=torch.int64, device=DEV), "Q": Q, "requests": table,
                "room": 4096 + int(3 * sum(r["nq"] * r["selectivity"] * case["m"] for r in reqs if r["kind"] == "eps"))}
    if op == "hist":
        f, h, w = case["frames"], case["h"], case["w"]
        base = torch.randint(0, 256, (f, -(-h // 24), -(-w // 24), 3), generator=g, device=DEV, dtype=torch.int16)
        frames = torch.empty(f, h, w, 3, dtype=torch.uint8, device=DEV)
        for i in range(f):   # blocks of one colour plus noise in [-6, 6]
            img = base[i].repeat_interleave(24, 0).repeat_interleave(24, 1)[:h, :w]
            img = img + torch.randint(-6, 7, img.shape, generator=g, device=DEV, dtype=torch.int16)
            frames[i] = img.clamp_(0, 255).to(torch.uint8)
        return {"op": op, "frames": frames, "boxes": torch.from_numpy(_boxes(case)).to(DEV), "bins": (case["bins"], 4, 4)}
    X = _views(g, _centres(g, max(1, case["n"] // VIEWS), case["d"]), case["n"], 0.01)
    return {"op": op, "ids": torch.arange(case["n"], dtype=torch.int64, device=DEV), "X": X,
            "eps": _threshold(X, None, "l2", case["per_row"])}


# ------------------------------------------------------------------------------- the calls

class _View:
    """A library-owned device array of n int64 values."""

    def __init__(self, ptr, n, owner):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<i8", "data": (ptr, False), "version": 2, "strides": None}


def _request_pairs(res, i):
    """Request i's pairs of a batch result, left on the device (dl_result_request_pairs)."""
    a, b, n = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_int64()
    rc = dl.load().dl_result_request_pairs(res._h, i, dl.DL_MEM_DEVICE, ctypes.byref(a), ctypes.byref(b), ctypes.byref(n))
    if rc != dl.DL_OK:
        raise dl.DLError(rc, dl.last_error())
    if n.value == 0:
        e = torch.empty(0, dtype=torch.int64, device=DEV)
        return e, e
    return tuple(torch.as_tensor(_View(p.value, n.value, res), device=DEV) for p in (a, b))


def _ordered(r, s, room):
    """The sorted pairs in a table of `room` entries, and their number."""
    out = torch.full((room,), -1, dtype=torch.int64, device=DEV)
    out[:len(r)] = torch.sort(torch.add(s, r, alpha=1 << 32)).values
    return [out, len(r)]


def _matrix(r, s, n, m):
    out = torch.zeros(n * m, dtype=torch.bool, device=DEV)
    return out.index_fill_(0, torch.add(s, r, alpha=m), True).view(n, m)


def run(state):
    op = state["op"]
    if op == "join":
        R, S = state["R"], state["S"]
        pairs = dl.sim_join(R, S, state["eps"], metric=state["metric"]).pairs_device()
        m = R.n if S is None else S.n
        return _matrix(*pairs, R.n, m) if R.n * m <= MATRIX else _ordered(*pairs, state["room"])
    if op == "pruned":
        return _ordered(*dl.sim_join(state["X"], None, state["eps"], prune=True).pairs_device(), state["room"])
    if op == "topk":
        return list(dl.topk_join(state["Q"], state["S"], state["k"], metric=state["metric"]).topk_host())
    if op == "batch":
        res = dl.batch_join(state["S"], state["ids"], state["Q"], state["requests"])
        pairs, near = [], []
        for i, r in enumerate(state["requests"]):
            if r["kind"] == "topk":
                near.append(res.request_topk(i))
            else:
                pairs.append(_request_pairs(res, i))
        out = {"ids": np.concatenate([a for a, _ in near]) if near else np.empty(0, np.int64),
               "dist2": np.concatenate([b for _, b in near]) if near else np.empty(0)}
        if pairs:
            out["pairs"] = _ordered(torch.cat([a for a, _ in pairs]), torch.cat([b for _, b in pairs]), state["room"])
        return out
    if op == "hist":
        return dl.color_hist(state["frames"], state["boxes"], state["bins"])
    comp, n = dl.dedup(dl.Store(state["ids"], state["X"]), state["eps"])
    return [comp, n]


# ------------------------------------------------------------------------------- work and exact values

def work(case):
    """Each operand row once (16-bit where the path contracts, else FP32), each result once; 2 d operations a pair."""
    op, d = case["op"], case.get("d", 0)
    if op == "join":
        n, m = case["n"], case["m"]
        pairs = n * m if m else n * (n - 1) // 2
        row = d * (4 if case["metric"] in ("l1", "chi2") else 2) + 8
        return {"bytes": (n + m) * row + 16 * n * case["per_row"], "flops": 2 * d * pairs}
    if op == "pruned":   # every row against its own object's 1,024 views
        n = case["n"]
        return {"bytes": n * (2 * d + 8) + 8 * n * case["per_row"], "flops": 2 * d * n * min(n, 1024) // 2}
    if op == "topk":
        n, m, k = case["n"], case["m"], case["k"]
        return {"bytes": (n + m) * d * (2 if case["metric"] == "l2" else 4) + 16 * n * k, "flops": 2 * d * n * m}
    if op == "batch":
        reqs, rows = _mix(case)
        m = case["m"]
        out = sum(r["nq"] * (r["selectivity"] * m if r["kind"] == "eps" else r["k"]) for r in reqs)
        return {"bytes": int(rows * d * 4 + m * d * 2 + 16 * out), "flops": 2 * d * rows * m}
    if op == "hist":
        b = _boxes(case).astype(np.int64)
        px = int(((b[:, 3] - b[:, 1]) * (b[:, 4] - b[:, 2])).sum())
        return {"bytes": 3 * px + 4 * len(b) * case["bins"] * 16, "flops": 4 * px}
    n = case["n"]
    return {"bytes": n * (4 * d + 16), "flops": d * n * (n - 1)}


def _exact_topk(Q, S, k, metric):
    """The k smallest distances of each row of Q to the rows of S, in 64 bits, ascending."""
    out = []
    S64 = S.double()
    if metric == "l2":
        sn = (S64 * S64).sum(1)
        for q in Q.double().split(64):
            d = (q * q).sum(1)[:, None] + sn[None, :] - 2.0 * (q @ S64.T)
            near = torch.topk(d, min(len(S), k + 28), dim=1, largest=False).indices   # then without cancellation
            t = torch.stack([(S64[near[i]] - q[i]).square_().sum(1) for i in range(len(q))])
            out.append(t.sort(1).values[:, :k])
    else:
        for q in Q.double():
            t = (q - S64).abs_()
            d = t.sum(1) if metric == "l1" else torch.where(q + S64 > 0, t * t / (q + S64), 0.0).sum(1)
            out.append(torch.topk(d, min(len(S), k), largest=False, sorted=True).values[None])
    v = torch.cat(out)
    if v.shape[1] < k:
        v = torch.cat([v, torch.full((len(v), k - v.shape[1]), -1.0, device=DEV, dtype=v.dtype)], 1)
    return v


def exact(case, seed):
    """Distances and histograms in 64 bits; pairs, ids and components are whole numbers."""
    g, op = _gen(seed), case["op"]
    if op == "topk":
        c = _centres(g, max(1, case["m"] // VIEWS), case["d"])
        S, Q = _views(g, c, case["m"], 0.01), _views(g, c, case["n"], 0.01)
        return [None, _exact_topk(Q, S, case["k"], case["metric"])]
    if op == "batch":
        reqs, rows = _mix(case)
        if not any(r["kind"] == "topk" for r in reqs):
            return None
        c = _centres(g, max(1, case["m"] // VIEWS), case["d"])
        S, Q = _views(g, c, case["m"], 0.01), _views(g, c, rows, 0.01)
        parts, at = [], 0
        for r in reqs:
            if r["kind"] == "topk":
                parts.append(_exact_topk(Q[at:at + r["nq"]], S, r["k"], "l2"))
            at += r["nq"]
        return {"ids": None, "dist2": torch.cat(parts), "pairs": None}
    if op == "hist":
        s = prepare(case, seed)
        b = s["bins"]
        n_bins = b[0] * b[1] * b[2]
        out = torch.empty(len(s["boxes"]), n_bins, dtype=torch.float64, device=DEV)
        for i, (f, x0, y0, x1, y1) in enumerate(s["boxes"].tolist()):
            p = s["frames"][f, y0:y1, x0:x1].reshape(-1, 3).long()
            j = ((p[:, 0] * b[0] // 256) * b[1] + p[:, 1] * b[1] // 256) * b[2] + p[:, 2] * b[2] // 256
            out[i] = torch.bincount(j, minlength=n_bins).double() / len(p)
        return out
    return None
