"""Timed cases of the D2-clustering framework: the calls of the C ABI that its
users make, through the Python binding, over the sizes of the repository's own
workload laws (paper_1302_0435_gb300/synth.py, bench.py, tests).

  pairs    d2_mallows_batch: distances of listed (bag, centroid) pairs
  round    one clustering round (Alg. 2 Steps 2-3*): set the centroids, assign
           with flows, move the supports, read the centroids back
  assign   d2_assign alone: nearest centroid of a batch
  all      d2_mallows_all: the certified distance of every (bag, centroid) pair
  table    d2_assign with symbol ground costs (the sequence variant)
  serve    a burst of host requests through the server
  level    d2_cluster_level: a whole hierarchical job
  weights  d2_update_weights: the joint weights of Alg. 1 Step 1

Inputs follow the laws of synth.py, drawn on the GPU so that large batches are
quick to make: every bag takes one mixture component, its supports scatter
around it, weights are Dirichlet, centroids follow the same law.
"""
import math

import torch

from paper_1302_0435_gb300 import d2

DEV = "cuda:0"

# Laws: support counts lo..hi (uneven: P(m) ~ m^-2), dimension, mixture
# components, element types, Dirichlet parameter (synth.py).
LAWS = {
    "plain": dict(lo=4, hi=8, d=3, comps=5, ldt="f64", wdt="f64", alpha=1.0),
    "image": dict(lo=8, hi=16, d=6, comps=32, ldt="f32", wdt="f32", alpha=0.5),
    "uneven": dict(lo=2, hi=64, d=16, comps=256, ldt="f32", wdt="f32", alpha=1.0),
    "high": dict(lo=16, hi=64, d=128, comps=1, ldt="bf16", wdt="f32", alpha=1.0),
    "serving": dict(lo=4, hi=64, d=32, comps=32, ldt="f32", wdt="f32", alpha=1.0),
}
TORCH = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
CODE = {"f64": d2.D2_F64, "f32": d2.D2_F32, "bf16": d2.D2_BF16}
SYMBOLS = 20


def listed():
    return [
        # a handful of distances on demand (nearest-neighbour re-ranking): latency of one call
        dict(name="pairs_few", kind="pairs", law="image", N=64, K=64, n=16, pairs=48),
        # a re-ranking batch over uneven bags, about a wave of warps
        dict(name="pairs_uneven", kind="pairs", law="uneven", N=2000, K=100, n=32, pairs=6000),
        # small FP64 data set, one clustering round: launches and waits count
        dict(name="round_plain_fp64", kind="round", law="plain", N=1000, K=8, n=8),
        # the image collection at full size, one round of the main loop
        dict(name="round_image", kind="round", law="image", N=200000, K=64, n=16),
        # every certified distance of the image collection (similarity tables, the metric)
        dict(name="all_image", kind="all", law="image", N=200000, K=64, n=16),
        # bags of very different sizes: nearest centroid of a large batch
        dict(name="assign_uneven", kind="assign", law="uneven", N=120000, K=256, n=32),
        # the same law, every distance; odd counts
        dict(name="all_uneven", kind="all", law="uneven", N=24001, K=255, n=32),
        # BF16 descriptors with wide bags: tensor-core ground costs, large trees
        dict(name="all_high_dim", kind="all", law="high", N=777, K=512, n=64),
        # histograms of symbol sequences under a substitution table
        dict(name="table_sequences", kind="table", law="sequence", N=40000, K=64, n=SYMBOLS),
        # a burst of requests on the server, one bag to a thousand
        dict(name="serve_burst", kind="serve", law="serving", K=1024, n=32,
             sizes="1,3,17,60,251,1000"),
        # the whole hierarchical job: segments, ten rounds each, merge
        dict(name="level_image", kind="level", law="image", N=60000, K=64, n=16, seg=5000,
             iters=10),
        # support weights of every cluster by the joint LP
        dict(name="weights_image", kind="weights", law="image", N=30000, K=64, n=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same calls and laws, sizes over their whole range."""
    kind = rng.choice(["pairs", "round", "assign", "all", "all", "table", "serve", "level",
                       "weights"])
    if kind == "pairs":
        law = rng.choice(["plain", "image", "uneven"])
        n = {"plain": 8, "image": 16, "uneven": 32}[law]
        return dict(kind=kind, law=law, N=_log(rng, 20, 3000), K=_log(rng, 8, 128),
                    n=rng.randint(max(2, n // 2), n), pairs=_log(rng, 5, 20000))
    if kind == "round":
        if rng.random() < 0.4:
            return dict(kind=kind, law="plain", N=_log(rng, 200, 20000), K=rng.randint(4, 16),
                        n=rng.randint(4, 8))
        return dict(kind=kind, law="image", N=_log(rng, 2000, 200000), K=rng.randint(16, 64),
                    n=rng.randint(8, 16))
    if kind == "assign":
        law = rng.choice(["image", "uneven", "high"])
        if law == "image":
            return dict(kind=kind, law=law, N=_log(rng, 500, 200000), K=rng.randint(8, 64),
                        n=rng.randint(8, 16))
        if law == "uneven":
            return dict(kind=kind, law=law, N=_log(rng, 500, 120000), K=rng.randint(32, 256),
                        n=rng.randint(16, 32))
        return dict(kind=kind, law=law, N=_log(rng, 50, 777), K=rng.randint(64, 512),
                    n=rng.randint(32, 64))
    if kind == "all":
        law = rng.choice(["image", "uneven", "high"])
        if law == "image":
            return dict(kind=kind, law=law, N=_log(rng, 500, 200000), K=rng.randint(8, 64),
                        n=rng.randint(8, 16))
        if law == "uneven":
            return dict(kind=kind, law=law, N=_log(rng, 500, 24000), K=rng.randint(32, 255),
                        n=rng.randint(16, 32))
        return dict(kind=kind, law=law, N=_log(rng, 50, 777), K=rng.randint(64, 512),
                    n=rng.randint(32, 64))
    if kind == "table":
        return dict(kind=kind, law="sequence", N=_log(rng, 500, 40000), K=rng.randint(8, 64),
                    n=SYMBOLS)
    if kind == "serve":
        sizes = [_log(rng, 1, 1000) for _ in range(rng.randint(1, 5))]
        return dict(kind=kind, law="serving", K=_log(rng, 128, 1024), n=rng.randint(16, 32),
                    sizes=",".join(map(str, sizes)))
    if kind == "level":
        K = rng.randint(16, 64)
        return dict(kind=kind, law="image", N=_log(rng, 4000, 60000), K=K, n=rng.randint(8, 16),
                    seg=_log(rng, 20 * K, 6000), iters=rng.randint(3, 10))
    return dict(kind=kind, law="image", N=_log(rng, 2000, 30000), K=rng.randint(16, 64),
                n=rng.randint(8, 16))


# ------------------------------------------------------------------ inputs --

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _offsets(sizes):
    off = torch.zeros(sizes.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(sizes, 0, out=off[1:])
    return off


def _sizes(g, law, N):
    if law == "uneven":
        p = torch.arange(2, 65, device=DEV, dtype=torch.float64) ** -2.0
        return torch.multinomial(p, N, replacement=True, generator=g) + 2
    s = LAWS[law]
    return torch.randint(s["lo"], s["hi"] + 1, (N,), device=DEV, generator=g)


def _means(g, law):
    s = LAWS[law]
    if law == "uneven":
        return 3.0 * torch.randn((s["comps"], s["d"]), device=DEV, generator=g)
    return 10.0 * torch.rand((s["comps"], s["d"]), device=DEV, generator=g) - 5.0


def _locs(g, law, sizes, means):
    s = LAWS[law]
    total = int(sizes.sum())
    x = torch.randn((total, s["d"]), device=DEV, generator=g,
                    dtype=torch.float64 if s["ldt"] == "f64" else torch.float32)
    if law == "high":  # nonnegative descriptors of unit length
        x = x.abs()
        x = x / x.norm(dim=1, keepdim=True)
    else:
        comp = torch.randint(0, means.shape[0], (sizes.numel(),), device=DEV, generator=g)
        x = x + means[torch.repeat_interleave(comp, sizes)].to(x.dtype)
    return x.to(TORCH[s["ldt"]]).contiguous()


def _weights(g, law, sizes):
    """Dirichlet(1) from exponentials, Dirichlet(1/2) from squared normals."""
    s = LAWS[law]
    total = int(sizes.sum())
    if s["alpha"] == 0.5:
        w = torch.randn(total, device=DEV, generator=g, dtype=torch.float64).square()
    else:
        w = torch.empty(total, device=DEV, dtype=torch.float64).exponential_(generator=g)
    tot = torch.segment_reduce(w, "sum", lengths=sizes)
    return (w / torch.repeat_interleave(tot, sizes)).to(TORCH[s["wdt"]])


def _ref(loc, w, off, ldt, wdt):
    count = off.shape[0] - 1
    top = int((off[1:] - off[:-1]).max())
    return d2.BagsRef(loc, w, off, count, loc.shape[1], CODE[ldt], CODE[wdt], top)


def _objects(g, law, N, means):
    s = LAWS[law]
    sizes = _sizes(g, law, N)
    return _ref(_locs(g, law, sizes, means), _weights(g, law, sizes), _offsets(sizes),
                s["ldt"], s["wdt"])


def _centroids(g, law, K, n, means):
    s = LAWS[law]
    sizes = torch.full((K,), n, dtype=torch.int64, device=DEV)
    w = torch.full((K * n,), 1.0 / n, dtype=TORCH[s["wdt"]], device=DEV)
    return _ref(_locs(g, law, sizes, means), w, _offsets(sizes), s["ldt"], s["wdt"])


def _histograms(g, count, profiles):
    """Symbol histograms of sequences of 100-600 symbols: the symbols present
    and their frequencies (FP32, one-dimensional symbol ids)."""
    cls = torch.randint(0, profiles.shape[0], (count,), device=DEV, generator=g)
    length = torch.randint(100, 601, (count, 1), device=DEV, generator=g)
    cnt = torch.poisson(profiles[cls] * length, generator=g)
    cnt[:, 0] += (cnt.sum(1) == 0)
    row, sym = torch.nonzero(cnt, as_tuple=True)
    freq = cnt[row, sym] / cnt.sum(1)[row]
    sizes = (cnt > 0).sum(1)
    return _ref(sym.to(torch.float32).reshape(-1, 1).contiguous(), freq.to(torch.float32),
                _offsets(sizes), "f32", "f32")


def _to_host(ref):
    loc, w, off = (x.cpu().numpy() for x in (ref.loc, ref.w, ref.off))
    return d2.BagsRef(loc, w, off, ref.s.count, ref.s.dim, ref.s.loc_dtype, ref.s.w_dtype,
                      ref.s.max_support)


def _inputs(case, seed):
    g = _gen(seed)
    if case["kind"] == "table":
        prof = torch.empty((3, SYMBOLS), device=DEV).exponential_(generator=g).square()
        prof = prof / prof.sum(1, keepdim=True)
        e = torch.randn((SYMBOLS, 6), device=DEV, generator=g, dtype=torch.float64)
        p = torch.exp(-torch.cdist(e, e).square() / 4.0)
        p = torch.log(p / p.sum(1, keepdim=True))
        cents = _histograms(g, case["K"], prof)
        return dict(objs=_histograms(g, case["N"], prof), cents=cents,
                    table=(-(p + p.T)).cpu().numpy())
    law = case["law"]
    means = _means(g, law)
    cents = _centroids(g, law, case["K"], case["n"], means)
    if case["kind"] == "serve":
        sizes = [int(x) for x in case["sizes"].split(",")]
        return dict(cents=cents, reqs=[_to_host(_objects(g, law, s, means)) for s in sizes])
    x = dict(cents=cents, objs=_objects(g, law, case["N"], means))
    if case["kind"] == "pairs":
        x["po"] = torch.randint(0, case["N"], (case["pairs"],), device=DEV, generator=g)
        x["pc"] = torch.randint(0, case["K"], (case["pairs"],), device=DEV, generator=g)
    if case["kind"] in ("round", "level", "weights"):
        x["omega"] = 0.5 + torch.rand(case["N"], device=DEV, generator=g, dtype=torch.float64)
    return x


def _empty(shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, device=DEV)


def _context():
    """A context with a clean status: reading it clears what it held when made."""
    ctx = d2.Context(0)
    try:
        d2.d2_sync(ctx)
    except d2.D2Error:
        pass
    return ctx


def prepare(case, seed):
    st = _inputs(case, seed)
    kind, K, n = case["kind"], case["K"], case["n"]
    ctx = st["ctx"] = _context()
    st["kind"], st["K"] = kind, K
    d2.d2_set_centroids(ctx, st["cents"])
    if kind == "serve":
        st["server"] = d2.Server(ctx, slots=8)
        return st
    if kind == "table":
        d2.d2_set_cost_table(ctx, st["table"])
    N, dim = st["objs"].count, st["objs"].s.dim
    if kind == "pairs":
        st["dist"] = _empty(case["pairs"])
        st["status"] = _empty(case["pairs"], torch.int32)
        return st
    st["labels"], st["dist"] = _empty(N, torch.int32), _empty(N)
    if kind == "all":
        st["all"] = _empty((N, K))
    elif kind == "round":
        stride = st["objs"].s.max_support + n - 1
        st["flows"] = (_empty((N, stride), torch.int32), _empty((N, stride)))
        st["eps"], st["loc"] = _empty(1), _empty((K * n, dim))
    elif kind == "level":
        st["loc"], st["mass"] = _empty((K * n, dim)), _empty(K)
        st["seg"], st["iters"] = case["seg"], case["iters"]
    elif kind == "weights":
        # the clusters whose weights are re-solved: every bag at its nearest centroid
        d2.d2_assign(ctx, st["objs"], st["labels"], st["dist"])
        d2.d2_sync(ctx)
        st["eps"], st["dim"] = _empty(K), dim
    return st


def run(st):
    ctx, kind = st["ctx"], st["kind"]
    if kind == "pairs":
        d2.d2_mallows_batch(ctx, st["objs"], st["po"], st["pc"], st["dist"], status=st["status"])
        return {"dist2": st["dist"], "status": st["status"]}
    if kind in ("assign", "table"):
        d2.d2_assign(ctx, st["objs"], st["labels"], st["dist"])
        return {"labels": st["labels"], "dist2": st["dist"]}
    if kind == "all":
        d2.d2_mallows_all(ctx, st["objs"], st["all"], st["labels"], st["dist"])
        return {"all": st["all"], "labels": st["labels"], "dist2": st["dist"]}
    if kind == "round":
        d2.d2_set_centroids(ctx, st["cents"])
        d2.d2_assign(ctx, st["objs"], st["labels"], st["dist"], omega=st["omega"], eps=st["eps"],
                     flows=st["flows"])
        d2.d2_update_locations(ctx, st["objs"], st["labels"], omega=st["omega"],
                               flows=st["flows"])
        d2.d2_get_centroids_into(ctx, st["loc"])
        return {"labels": st["labels"], "dist2": st["dist"], "eps": st["eps"], "loc": st["loc"]}
    if kind == "level":
        d2.d2_cluster_level(ctx, st["objs"], st["K"], st["seg"], st["iters"], st["loc"],
                            st["mass"], st["labels"], omega=st["omega"])
        return {"loc": st["loc"], "mass": st["mass"], "labels": st["labels"]}
    if kind == "weights":
        d2.d2_set_centroids(ctx, st["cents"])
        d2.d2_update_weights(ctx, st["objs"], st["labels"], omega=st["omega"], eps=st["eps"])
        return {"weights": d2.d2_get_centroids(ctx, st["dim"])[1], "eps": st["eps"]}
    tickets = [st["server"].submit(r) for r in st["reqs"]]
    out = {}
    for k, t in enumerate(tickets):
        _, lab, dist, _ = st["server"].poll(t)
        out["labels%d" % k], out["dist2_%d" % k] = lab, dist
    return out


# -------------------------------------------------------------------- work --

def work(case):
    """Each input read once and each output written once; operations: the
    ground costs of the pairs that are solved and one reduced-cost check of
    each cell (the proof of optimality).  Where only the nearest centroid is
    asked for, one pair per bag is solved and the others are told apart by
    the distance of the means."""
    kind, K, n = case["kind"], case["K"], case["n"]
    if kind == "table":
        m, d, lb, wb = 15.0, 1, 4, 4
    else:
        s = LAWS[case["law"]]
        m = 5.9 if case["law"] == "uneven" else (s["lo"] + s["hi"]) / 2.0
        d, wb = s["d"], 8 if s["wdt"] == "f64" else 4
        lb = {"f64": 8, "f32": 4, "bf16": 2}[s["ldt"]]
    N = sum(int(x) for x in case["sizes"].split(",")) if kind == "serve" else case["N"]
    pair = m * n * (3.0 * d + 2.0)
    inputs = N * (m * (d * lb + wb) + 8.0) + K * n * (d * lb + wb)
    moments = 3.0 * d * (N * m + K * n) + 3.0 * d * N * K
    if kind == "pairs":
        bags = min(case["pairs"], N)
        return {"bytes": bags * (m * (d * lb + wb) + 8.0) + K * n * (d * lb + wb)
                + case["pairs"] * 28.0, "flops": case["pairs"] * pair}
    if kind == "all":
        return {"bytes": inputs + 8.0 * N * K + 12.0 * N, "flops": N * K * pair}
    if kind in ("assign", "table", "serve"):
        return {"bytes": inputs + 12.0 * N, "flops": moments + N * pair}
    if kind == "round":
        flows = 12.0 * N * (m + n - 1)
        return {"bytes": inputs + 20.0 * N + 2.0 * flows + 8.0 * K * n * d,
                "flops": moments + N * pair + 2.0 * N * (m + n - 1) * (d + 1)}
    if kind == "level":
        top = -(-N // case["seg"]) * K if N > case["seg"] else 0
        rounds = case["iters"] * (N + top)
        one = 3.0 * d * (m + K) + pair + 2.0 * (m + n - 1) * (d + 1)
        return {"bytes": inputs + 12.0 * N + 8.0 * K * n * d, "flops": rounds * one}
    return {"bytes": inputs + 12.0 * N + 8.0 * K * (n + 1), "flops": N * pair}


# ------------------------------------------------------------------- exact --

def _transport(C, p, q):
    """Transportation LPs min <C, w> with row sums p and column sums q, in
    64 bits: C [B, m, n].  Revised simplex from the northwest corner, the
    most negative reduced cost entering; the last column's constraint is
    dropped.  Returns the optimal w [B, m, n]."""
    B, m, n = C.shape
    R = m + n - 1
    idx = torch.arange(B, device=C.device)
    a = torch.zeros(B, dtype=torch.int64, device=C.device)
    r = torch.zeros_like(a)
    rows, cols = [], []
    P, Q = p.cumsum(1), q.cumsum(1)
    for _ in range(R):  # the staircase: down when the row's mass is used up first
        rows.append(a.clone())
        cols.append(r.clone())
        down = ((P[idx, a] <= Q[idx, r]) & (a < m - 1)) | (r == n - 1)
        a = a + down
        r = r + (~down).long()
        a.clamp_(max=m - 1)
        r.clamp_(max=n - 1)
    ba, br = torch.stack(rows, 1), torch.stack(cols, 1)
    A = torch.zeros((B, m + n, R), dtype=C.dtype, device=C.device)
    one = torch.ones((B, 1, R), dtype=C.dtype, device=C.device)
    A.scatter_(1, ba[:, None, :], one)
    A.scatter_(1, (m + br)[:, None, :], one)
    inv = torch.linalg.inv(A[:, :R, :])
    b = torch.cat([p, q], 1)[:, :R]
    x = torch.einsum("bij,bj->bi", inv, b)
    tol = 1e-13 * C.amax(dim=(1, 2))
    for _ in range(50 * R):
        y = torch.einsum("bi,bij->bj", C[idx[:, None], ba, br], inv)
        v = torch.cat([y[:, m:], torch.zeros((B, 1), dtype=C.dtype, device=C.device)], 1)
        red = (C - y[:, :m, None] - v[:, None, :]).reshape(B, m * n)
        best, cell = red.min(1)
        act = best < -tol
        if not bool(act.any()):
            break
        ea, er = cell // n, cell % n
        col = inv[idx, :, ea] + torch.where((er < n - 1)[:, None],
                                            inv[idx, :, m + er.clamp(max=n - 2)], 0.0)
        ratio = torch.where(col > 0.5, x.clamp(min=0.0) / col, torch.inf)
        th, out = ratio.min(1)
        th = torch.where(act, th, 0.0)
        piv = inv[idx, out]
        sel = torch.zeros_like(col).scatter_(1, out[:, None], 1.0)
        col = torch.where(act[:, None], col - sel, 0.0)  # pivots of a spanning tree are 1
        x = x - th[:, None] * col
        x[idx, out] = torch.where(act, th, x[idx, out])
        inv = inv - col[:, :, None] * piv[:, None, :]
        ba[idx, out] = torch.where(act, ea, ba[idx, out])
        br[idx, out] = torch.where(act, er, br[idx, out])
    w = torch.zeros((B, m * n), dtype=C.dtype, device=C.device)
    w.scatter_add_(1, ba * n + br, x)
    return w.reshape(B, m, n)


def _exact_pairs(objs, cents, n, po, pc):
    """D^2 and the flows (object support, centroid support, mass) of listed pairs."""
    loc, w, off = objs.loc.double(), objs.w.double(), objs.off
    dim = objs.s.dim
    cl = cents.loc.double().reshape(-1, n, dim)
    cw = cents.w.double().reshape(-1, n)
    cw = cw / cw.sum(1, keepdim=True)
    size = (off[1:] - off[:-1])[po]
    dist = torch.zeros(po.numel(), dtype=torch.float64, device=DEV)
    moves = []
    for m in torch.unique(size).tolist():
        for part in torch.split(torch.nonzero(size == m).reshape(-1), 1 << 14):
            rows = off[po[part]][:, None] + torch.arange(m, device=DEV)
            x, p = loc[rows], w[rows]
            p = p / p.sum(1, keepdim=True)
            y = cl[pc[part]]
            C = (x[:, :, None, :] - y[:, None, :, :]).square().sum(-1)
            flow = _transport(C, p, cw[pc[part]])
            dist[part] = (flow * C).sum(dim=(1, 2))
            moves.append((part, rows, flow))
    return dist, moves


def exact(case, seed):
    """Distances (and a small round's labels and centroids) by a batched
    transportation simplex in 64 bits.  Batches of more pairs, and results
    whose own arithmetic is a stopping rule, have no such value."""
    kind = case["kind"]
    if kind == "pairs" and case["pairs"] <= 8000:
        x = _inputs(case, seed)
        dist, _ = _exact_pairs(x["objs"], x["cents"], case["n"], x["po"], x["pc"])
        return {"dist2": dist, "status": None}
    if kind == "round" and case["N"] * case["K"] <= 40000:
        x = _inputs(case, seed)
        N, K, n, dim = case["N"], case["K"], case["n"], x["objs"].s.dim
        po = torch.arange(N, device=DEV).repeat_interleave(K)
        pc = torch.arange(K, device=DEV).repeat(N)
        dist, moves = _exact_pairs(x["objs"], x["cents"], n, po, pc)
        best, lab = dist.reshape(N, K).min(1)
        num = torch.zeros((K * n, dim), dtype=torch.float64, device=DEV)
        den = torch.zeros(K * n, dtype=torch.float64, device=DEV)
        for part, rows, flow in moves:
            mine = torch.nonzero(lab[po[part]] == pc[part]).reshape(-1)
            f = flow[mine] * x["omega"][po[part[mine]]][:, None, None]
            at = (pc[part[mine]] * n)[:, None] + torch.arange(n, device=DEV)
            num.index_add_(0, at.reshape(-1), torch.einsum(
                "bmn,bmd->bnd", f, x["objs"].loc.double()[rows[mine]]).reshape(-1, dim))
            den.index_add_(0, at.reshape(-1), f.sum(1).reshape(-1))
        old = x["cents"].loc.double()
        loc = torch.where(den[:, None] > 0, num / den.clamp(min=1e-300)[:, None], old)
        if LAWS[case["law"]]["ldt"] != "f64":
            loc = loc.to(TORCH[LAWS[case["law"]]["ldt"]]).double()
        return {"labels": None, "dist2": best, "eps": (x["omega"] * best).sum().reshape(1),
                "loc": loc}
    return None
