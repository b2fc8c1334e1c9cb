"""The calls whose time is measured: what a user of the framework has it do,
through its public Python entry points, from a single interactive query to the
largest batch, with the values of each call in 64-bit arithmetic beside it.

A case is a dict of plain values; its "kind" names the entry point:
  search  : Database.search (query prep, PartialReduce, ExactRescoring, FP32 re-rank)
  exact   : Database.search_exact (ground truth)
  partial : Database.partial_reduce (Alg. 1 alone)
  amk     : approx_max_k on a score matrix the caller holds
  train   : knn_topk forward and backward, gradients of queries and rows
  build   : Database(...) from FP32 rows
"""
import math

import torch

from paper_2206_14286_gb300 import search as S
from paper_2206_14286_gb300 import synth
from paper_2206_14286_gb300.autograd import knn_topk

_ESZ = {"f32": 4, "bf16": 2, "e4m3": 1, "e4m3t": 1}


def listed():
    return [
        # one interactive query against the 1M x 128 database: latency
        dict(name="query_one", kind="search", metric="l2", dtype="bf16", N=1_000_000, D=128, M=1,
             K=10, L=0, recall=0.95, rerank=2, bins="mod", centres=256),
        # the plain FP32 workload: a small database that fits in cache, the
        # smallest call in bytes and operations
        dict(name="f32_16k", kind="search", metric="ip", dtype="f32", N=16_384, D=128, M=64, K=10,
             L=1024, recall=0.95, rerank=1, bins="mod", centres=0),
        # the headline batch: 1024 queries on 1M x 128 rows
        dict(name="batch_l2_1m", kind="search", metric="l2", dtype="bf16", N=1_000_000, D=128,
             M=1024, K=10, L=0, recall=0.95, rerank=2, bins="mod", centres=256),
        # a serving batch on the long-row database of the serving loop
        dict(name="serve_ip_4m", kind="search", metric="ip", dtype="bf16", N=4_000_000, D=768,
             M=64, K=100, L=0, recall=0.95, rerank=2, bins="mod", centres=256),
        # contiguous bins with odd sizes everywhere
        dict(name="runs_odd", kind="search", metric="l2", dtype="bf16", N=700_001, D=100, M=333,
             K=20, L=0, recall=0.97, rerank=2, bins="contiguous", centres=256),
        # the FP8 workload with per-row scales: the largest call
        dict(name="cos_e4m3_10m", kind="search", metric="cos", dtype="e4m3", N=10_000_000, D=96,
             M=10_000, K=100, L=8192, recall=0.95, rerank=8, bins="mod", centres=1024),
        # the same path with one database-wide scale, a fifth of the rows and queries
        dict(name="cos_e4m3t_2m", kind="search", metric="cos", dtype="e4m3t", N=2_000_000, D=96,
             M=2000, K=100, L=8192, recall=0.95, rerank=8, bins="mod", centres=1024),
        # exact FP32 search: the ground truth a recall measurement needs
        dict(name="exact_f32", kind="exact", metric="l2", dtype="f32", N=1_000_000, D=128, M=100,
             K=10, centres=256),
        # the operator on a BF16 score matrix a GEMM has written
        dict(name="amk_bf16_1m", kind="amk", dtype="bf16", M=1024, N=1_000_000, K=10, L=0,
             recall=0.95, bins="mod", is_min=False, aggregate=True),
        # approx_min_k on an FP32 distance matrix with odd sizes
        dict(name="amk_f32_odd", kind="amk", dtype="f32", M=250, N=100_003, K=100, L=0,
             recall=0.95, bins="mod", is_min=True, aggregate=True),
        # a training step through the differentiable search
        dict(name="train_ip_1m", kind="train", metric="ip", dtype="bf16", N=1_000_000, D=256,
             M=4096, K=32, L=0, recall=0.95),
        # building a cosine FP8 database from FP32 rows
        dict(name="build_cos_2m", kind="build", metric="cos", dtype="e4m3", N=2_000_000, D=96,
             centres=1024),
    ]


# ---------------------------------------------------------------------------
# Drawn cases
# ---------------------------------------------------------------------------
def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_one(rng):
    kind = rng.choice(["search", "search", "search", "search", "exact", "partial", "amk", "amk",
                       "train", "build"])
    if kind == "search":
        dtype = rng.choice(["bf16", "bf16", "f32", "e4m3", "e4m3t"])
        metric = rng.choice(["ip", "l2", "cos"])
        D = _log(rng, 16, 1024 if dtype == "bf16" else 256)
        runs = dtype == "bf16" and rng.random() < 0.25
        return dict(kind=kind, metric=metric, dtype=dtype,
                    N=_log(rng, 10_000, 1_000_000 if dtype == "f32" else 4_000_000), D=D,
                    M=_log(rng, 1, 10_000), K=_log(rng, 1, 100), L=0,
                    recall=round(rng.uniform(0.9, 0.99), 3),
                    rerank=8 if dtype.startswith("e4m3") else rng.choice([1, 2, 4]),
                    bins="contiguous" if runs else "mod", centres=256)
    if kind == "exact":
        return dict(kind=kind, metric=rng.choice(["ip", "l2", "cos"]),
                    dtype=rng.choice(["f32", "f32", "bf16"]), N=_log(rng, 10_000, 1_000_000),
                    D=_log(rng, 16, 256), M=_log(rng, 1, 512), K=_log(rng, 1, 100), centres=256)
    if kind == "partial":
        return dict(kind=kind, metric=rng.choice(["ip", "l2"]), dtype=rng.choice(["bf16", "f32"]),
                    N=_log(rng, 10_000, 1_000_000), D=_log(rng, 16, 512), M=_log(rng, 1, 1024),
                    L=_log(rng, 64, 4096), bins="mod", centres=256)
    if kind == "amk":
        return dict(kind=kind, dtype=rng.choice(["bf16", "f32"]), M=_log(rng, 1, 1024),
                    N=_log(rng, 1000, 1_000_000), K=_log(rng, 1, 100), L=0,
                    recall=round(rng.uniform(0.9, 0.99), 3), bins=rng.choice(["mod", "contiguous"]),
                    is_min=rng.random() < 0.5, aggregate=rng.random() < 0.75)
    if kind == "train":
        return dict(kind=kind, metric=rng.choice(["ip", "l2"]), dtype="bf16",
                    N=_log(rng, 50_000, 1_000_000), D=_log(rng, 32, 256), M=_log(rng, 16, 4096),
                    K=_log(rng, 1, 32), L=0, recall=0.95)
    return dict(kind=kind, metric=rng.choice(["l2", "cos", "ip"]),
                dtype=rng.choice(["bf16", "e4m3", "e4m3t", "f32"]), N=_log(rng, 10_000, 1_500_000),
                D=_log(rng, 16, 512), centres=256)


def _seconds(c):
    """A rough time of one pass, to keep the drawn cases below the largest listed one."""
    w = work(c)
    rate = 1.5e13 if c["dtype"] == "f32" else 4e14
    t = w["flops"] / rate + w["bytes"] / 2e12
    if c["kind"] == "exact":
        t += c["M"] * c["N"] / 5e10
    if c["kind"] == "build":
        t += c["N"] * c["D"] / 1e10
    return t


def draw(rng):
    while True:
        c = _draw_one(rng)
        N, L, K = c["N"], _bins(c), c.get("K", 1)
        if K <= L <= N and _seconds(c) <= 0.012 and N * c.get("D", 1) <= 1_500_000_000:
            return c


# ---------------------------------------------------------------------------
# Inputs and the call
# ---------------------------------------------------------------------------
def _bins(c):
    """L of the case: as given, or the smallest with ((L-1)/L)^(K-1) >= recall (Eq. 13-14)."""
    if c.get("L"):
        return c["L"]
    K, r = c.get("K", 1), c.get("recall", 0.95)
    if K <= 1:
        return 1
    L = max(1, math.ceil(1.0 / (1.0 - r ** (1.0 / (K - 1)))))
    law = lambda n: (1.0 - 1.0 / n) ** (K - 1)  # noqa: E731
    while L > 1 and law(L - 1) >= r:
        L -= 1
    while law(L) < r:
        L += 1
    return min(L, c["N"])


def _rows(c, seed):
    """(database rows, query rows) of the case, FP32 on the GPU."""
    dev = torch.device("cuda")
    N, D, M, nc = c["N"], c["D"], c.get("M", 0), c.get("centres", 0)
    if nc:
        x = synth.mixture_device(N, D, nc, 2 * seed, dev, centre_seed=seed)
        q = synth.mixture_device(M, D, nc, 2 * seed + 1, dev, centre_seed=seed) if M else None
        return x, q
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    std = 1.0 / math.sqrt(D) if c["kind"] == "train" else 1.0
    x = torch.randn((N, D), generator=g, device=dev) * std
    q = torch.randn((M, D), generator=g, device=dev) * std if M else None
    return x, q


def _scores(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    s = torch.empty((c["M"], c["N"]), dtype=torch.bfloat16 if c["dtype"] == "bf16" else torch.float32,
                    device="cuda")
    step = max(1, (1 << 27) // c["N"])
    for i in range(0, c["M"], step):
        e = min(c["M"], i + step)
        s[i:e] = torch.randn((e - i, c["N"]), generator=g, device="cuda")
    return s


def _targets(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) + (1 << 40))
    return torch.randn((c["M"], c["K"]), generator=g, device="cuda")


def prepare(case, seed):
    c, seed = case, int(seed)
    if c["kind"] == "amk":
        return dict(case=c, scores=_scores(c, seed))
    x, q = _rows(c, seed)
    if c["kind"] == "build":
        return dict(case=c, x=x)
    db = S.Database(x, metric=c["metric"], dtype=c["dtype"])
    if c["kind"] == "train":
        return dict(case=c, db=db, x=x.requires_grad_(), q=q.requires_grad_(),
                    t=_targets(c, seed))
    return dict(case=c, db=db, q=q)


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "search":
        val, idx = state["db"].search(state["q"], c["K"], L=c["L"] or None,
                                      recall_target=c["recall"], rerank=c["rerank"],
                                      bins=c["bins"])
        return {"val": val, "idx": idx}
    if kind == "exact":
        val, idx = state["db"].search_exact(state["q"], c["K"])
        return {"val": val, "idx": idx}
    if kind == "partial":
        val, idx = state["db"].partial_reduce(state["q"], c["L"], bins=c["bins"])
        return {"val": val, "idx": idx}
    if kind == "amk":
        val, idx = S.approx_max_k(state["scores"], c["K"], L=c["L"] or None,
                                  recall_target=c["recall"], bins=c["bins"], is_min=c["is_min"],
                                  aggregate_to_topk=c["aggregate"])
        return {"val": val, "idx": idx}
    if kind == "train":
        q, x = state["q"], state["x"]
        val, idx = knn_topk(q, x, state["db"], c["K"], recall_target=c["recall"])
        loss = (torch.softmax(val, 1) * state["t"]).sum()
        dq, dx = torch.autograd.grad(loss, (q, x))
        return {"val": val.detach(), "idx": idx, "dq": dq, "dx": dx}
    db = S.Database(state["x"], metric=c["metric"], dtype=c["dtype"])
    out = {"lp": db.lp}
    if db.scale is not None:
        out["scale"] = db.scale
    if db.hnorm is not None:
        out["hnorm"] = db.hnorm
    if c["metric"] == "cos":
        out["f32"] = db.f32
    return out


def work(case):
    """Bytes: every input read once, every result written once (the FP32 rows of the
    re-rank counted once per candidate, at most the whole database). FLOPs: of the
    contraction, and of the gradients' two gathers."""
    c = case
    kind, N = c["kind"], c["N"]
    if kind == "amk":
        width = c["K"] if c["aggregate"] else _bins(c)
        return {"bytes": c["M"] * N * _ESZ[c["dtype"]] + c["M"] * width * 8, "flops": 0}
    D, M = c["D"], c.get("M", 0)
    pitch = (D + 15) // 16 * 16
    side = (4 * N if c["metric"] == "l2" else 0) + (4 * N if c["dtype"].startswith("e4m3") else 0)
    lp = N * pitch * _ESZ[c["dtype"]]
    if kind == "build":
        return {"bytes": N * D * 4 + lp + side + (N * D * 4 if c["metric"] == "cos" else 0),
                "flops": 0}
    flops = 2 * M * N * D
    b = N * D * _ESZ[c["dtype"]] + side + M * D * 4
    if kind == "partial":
        return {"bytes": b + M * c["L"] * 8, "flops": flops}
    K = c["K"]
    b += M * K * 8
    if kind == "exact":
        return {"bytes": b, "flops": flops}
    cand = M * min(c.get("rerank", 2) * K, _bins(c))
    b += min(cand, N) * D * 4
    if kind == "train":
        b += M * K * D * 4 + M * K * 8 + 2 * M * D * 4 + N * D * 4
        flops += 4 * M * K * D
    return {"bytes": b, "flops": flops}


# ---------------------------------------------------------------------------
# The same results in 64-bit arithmetic
# ---------------------------------------------------------------------------
def _unit(x):
    x = x.double()
    n = x.norm(dim=1, keepdim=True)
    return x / torch.where(n == 0, torch.ones_like(n), n)


def _codes(y, dtype, whole):
    """(values as the contraction sees them, E4M3 codes' scale) of FP32 rows y."""
    if dtype == "f32":
        return y.double(), None
    if dtype == "bf16":
        return y.to(torch.bfloat16).double(), None
    mx = y.abs().amax() if whole else y.abs().amax(dim=1)
    s = torch.where(mx > 0, mx / 448.0, torch.ones_like(mx))
    s = s.expand(y.shape[0]).contiguous()
    return (y / s[:, None]).to(torch.float8_e4m3fn).double() * s[:, None].double(), s


def _stored(x, c, whole):
    """FP64 values of the rows as stored for the contraction."""
    y = _unit(x).float() if c["metric"] == "cos" else x
    return _codes(y, c["dtype"], whole)[0]


def _score(qs, xs, metric):
    s = qs @ xs.t()
    return s - 0.5 * (xs * xs).sum(1)[None, :] if metric == "l2" else s


def _bin_best(score_rows, M, N, L, bins):
    """Best score and row of every bin; score_rows(a, b): M x (b - a) scores of rows a..b-1."""
    V = torch.full((M, L), -math.inf, dtype=torch.float64, device="cuda")
    A = torch.full((M, L), -1, dtype=torch.int64, device="cuda")
    room = max(1, (1 << 27) // max(M, 1))

    def take(a, rows, width, b0, by_bin):
        # rows x width scores: width bins side by side, or rows bins one after another
        s = score_rows(a, a + rows * width).reshape(M, rows, width)
        v, k = s.max(dim=2 if by_bin else 1)
        n = v.shape[1]
        at = torch.arange(n, device="cuda")[None, :]
        j = a + (at * width + k if by_bin else k * width + at)
        better = v > V[:, b0:b0 + n]
        V[:, b0:b0 + n] = torch.where(better, v, V[:, b0:b0 + n])
        A[:, b0:b0 + n] = torch.where(better, j, A[:, b0:b0 + n])

    if bins == "mod":
        T, step = N // L, max(1, room // L)
        for t in range(0, T, step):
            take(t * L, min(step, T - t), L, 0, False)
        if N % L:
            take(T * L, 1, N % L, 0, False)
    else:
        q, r = N // L, N % L
        for width, first, count, a0 in ((q + 1, 0, r, 0), (q, r, L - r, r * (q + 1))):
            step = max(1, room // width)
            for b in range(0, count, step):
                take(a0 + b * width, min(step, count - b), width, first + b, True)
    return V, A


def _values(q, x, idx, metric):
    """FP64 reported values of rows idx for each query."""
    out = torch.empty(idx.shape, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 27) // (idx.shape[1] * q.shape[1]))
    for i in range(0, q.shape[0], step):
        rows = x[idx[i:i + step]].double()
        a = q[i:i + step, None, :].double()
        if metric == "cos":
            a = a / a.norm(dim=2, keepdim=True)
            rows = rows / rows.norm(dim=2, keepdim=True)
        out[i:i + step] = ((a - rows) ** 2).sum(2) if metric == "l2" else (a * rows).sum(2)
    return out


def _best_rows(x, q, c, L, bins, Kp, K):
    """(values, rows) of the bin-wise search with a re-rank of Kp, best first."""
    qs = _stored(q, c, False)
    whole = c["dtype"] == "e4m3t"
    scale_x = None
    if whole:
        y = x if c["metric"] != "cos" else None
        top = max(float(((_unit(x[a:a + (1 << 18)]).float()) if y is None else x[a:a + (1 << 18)])
                        .abs().amax()) for a in range(0, c["N"], 1 << 18))
        scale_x = torch.tensor(top, device="cuda") / 448.0

    def rows(a, b):
        if not whole:
            return _stored(x[a:b], c, False)
        y = _unit(x[a:b]).float() if c["metric"] == "cos" else x[a:b]
        return (y / scale_x).to(torch.float8_e4m3fn).double() * scale_x.double()

    V, A = _bin_best(lambda a, b: _score(qs, rows(a, b), c["metric"]), c["M"], c["N"], L, bins)
    cand = A.gather(1, V.topk(Kp, dim=1).indices)
    val = _values(q, x, cand, c["metric"])
    at = val.topk(K, dim=1, largest=c["metric"] != "l2").indices
    return val.gather(1, at), cand.gather(1, at)


def exact(case, seed):
    c, seed = case, int(seed)
    kind = c["kind"]
    if kind not in ("amk", "build") and 2 * c["M"] * c["N"] * c["D"] > 5e12:
        return None
    if kind == "amk":
        s = _scores(c, seed)
        s = -s if c["is_min"] else s
        V, _ = _bin_best(lambda a, b: s[:, a:b].double(), c["M"], c["N"], _bins(c), c["bins"])
        if c["aggregate"]:
            V = V.topk(c["K"], dim=1).values
        return {"val": -V if c["is_min"] else V, "idx": None}
    x, q = _rows(c, seed)
    if kind == "build":
        out = {"lp": None}
        y = torch.cat([_unit(x[a:a + (1 << 20)]) for a in range(0, c["N"], 1 << 20)]) \
            if c["metric"] == "cos" else x.double()
        if c["dtype"].startswith("e4m3"):
            mx = y.abs().amax().expand(c["N"]) if c["dtype"] == "e4m3t" else y.abs().amax(dim=1)
            out["scale"] = mx / 448.0
        if c["metric"] == "l2":
            if c["dtype"] == "e4m3t":
                s = (x.abs().amax() / 448.0)
                st = (x / s).to(torch.float8_e4m3fn).double() * s.double()
            else:
                st = _codes(x, c["dtype"], False)[0]
            out["hnorm"] = 0.5 * (st * st).sum(1)
        if c["metric"] == "cos":
            out["f32"] = y
        return out
    if kind == "partial":
        qs = _stored(q, c, False)
        V, _ = _bin_best(lambda a, b: _score(qs, _stored(x[a:b], c, False), c["metric"]), c["M"],
                         c["N"], c["L"], c["bins"])
        return {"val": V, "idx": None}
    K = c["K"]
    if kind == "exact":
        # every row its own bin: the best K scores, chunk by chunk
        qs, best, at = _stored(q, c, False), None, None
        step = max(K, (1 << 27) // c["M"])
        for a in range(0, c["N"], step):
            b = min(c["N"], a + step)
            v, k = _score(qs, _stored(x[a:b], c, False), c["metric"]).topk(min(K, b - a), dim=1)
            best = v if best is None else torch.cat([best, v], 1)
            at = k + a if at is None else torch.cat([at, k + a], 1)
            best, o = best.topk(min(K, best.shape[1]), dim=1)
            at = at.gather(1, o)
        val = _values(q, x, at, c["metric"])
        return {"val": val.sort(dim=1, descending=c["metric"] != "l2").values, "idx": None}
    L = _bins(c)
    Kp = max(K, min(c.get("rerank", 2) * K, L))
    val, idx = _best_rows(x, q, c, L, c.get("bins", "mod"), Kp, K)
    if kind == "search":
        return {"val": val, "idx": None}
    # the gradients of the loss with respect to the values, the queries and the rows
    t = _targets(c, seed).double()
    p = torch.softmax(val, 1)
    g = p * (t - (p * t).sum(1, keepdim=True))
    xd, qd = x.double(), q.double()
    rows = xd[idx]
    dx = torch.zeros_like(xd)
    if c["metric"] == "l2":
        diff = qd[:, None, :] - rows
        dq = (2.0 * g[:, :, None] * diff).sum(1)
        dx.index_add_(0, idx.reshape(-1), (-2.0 * g[:, :, None] * diff).reshape(-1, c["D"]))
    else:
        dq = (g[:, :, None] * rows).sum(1)
        dx.index_add_(0, idx.reshape(-1), (g[:, :, None] * qd[:, None, :]).reshape(-1, c["D"]))
    return {"val": val, "idx": None, "dq": dq, "dx": dx}
