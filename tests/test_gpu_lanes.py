"""The screen that runs several pairs per warp, at the edges of its shapes.

A launch's row bound picks the lanes per pair and the node slots per lane, the
centroid bound the column lanes, so the sizes are the bounds of every shape and
their neighbours, in one launch (small batch) and cut into bins (large batch).
Every D^2 is certified within 2^-24 D^2 + 2^-43 c_max of the optimum, so the
oracle's values may differ by 1e-7 relative plus 1e-12 of the largest cost.
"""
import numpy as np
import pytest

from paper_1302_0435_gb300.synth import Bags

pytestmark = pytest.mark.gpu

EDGES = [1, 2, 4, 5, 8, 9, 12, 13, 16, 17, 24, 25, 32, 33, 48, 49, 63, 64]


@pytest.fixture(scope="module")
def d2():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_0435_gb300 import build, d2 as mod
    build.build()
    mod.load()
    return mod


def bags(rng, sizes, d, law):
    """normal: scattered supports; lattice: integer supports and weights
    (equal costs, zero and equal masses); far: bags far apart."""
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    T = int(off[-1])
    if law == "lattice":
        loc = rng.integers(0, 3, size=(T, d)).astype(np.float32)
        w = rng.integers(0, 3, size=T).astype(np.float32)
        w[off[:-1]] += 1.0
    else:
        loc = rng.normal(size=(T, d)).astype(np.float32)
        if law == "far":
            loc += np.repeat(rng.normal(0, 20, size=(len(sizes), d)), sizes, axis=0).astype(np.float32)
        w = rng.exponential(size=T).astype(np.float32)
    return Bags(loc, w, off, "f32", "f32")


def run_all(d2, objs, cents):
    import torch
    ctx = d2.Context(0)
    d2.d2_set_centroids(ctx, d2.bags_from_synth(cents, device="cuda:0"))
    ob = d2.bags_from_synth(objs, device="cuda:0")
    N, K = objs.count, cents.count
    every = torch.empty((N, K), dtype=torch.float64, device="cuda:0")
    lab = torch.empty(N, dtype=torch.int32, device="cuda:0")
    dist = torch.empty(N, dtype=torch.float64, device="cuda:0")
    assert d2.d2_mallows_all(ctx, ob, every, lab, dist) == d2.D2_OK
    d2.d2_sync(ctx)
    lab2, dist2 = torch.empty_like(lab), torch.empty_like(dist)
    assert d2.d2_assign(ctx, ob, lab2, dist2) == d2.D2_OK
    d2.d2_sync(ctx)
    ctx.close()
    return [t.cpu().numpy() for t in (every, lab, dist, lab2, dist2)]


def check(oracle_mod, objs, cents, out, rows):
    every, lab, dist, lab2, dist2 = out
    sub = objs.subset(rows)
    _, _, ref = oracle_mod.assign(sub, cents, nthreads=8, return_all=True)
    big = float(np.max(np.abs(objs.loc))) + float(np.max(np.abs(cents.loc)))
    floor = 1e-12 * objs.dim * big * big
    assert np.all(np.abs(every[rows] - ref) <= 1e-7 * ref + floor)
    for l, dd in ((lab, dist), (lab2, dist2)):
        at = ref[np.arange(len(rows)), l[rows]]
        assert np.all(at <= ref.min(axis=1) * (1 + 1e-9) + floor)
        assert np.all(np.abs(dd[rows] - at) <= 1e-7 * at + floor)


@pytest.mark.parametrize("law", ["normal", "lattice", "far"])
@pytest.mark.parametrize("n,d", [(1, 3), (4, 6), (15, 6), (16, 16), (17, 5), (20, 1), (32, 32),
                                 (33, 3), (64, 8)])
def test_shapes(d2, oracle_mod, n, d, law):
    rng = np.random.default_rng(1000 * n + d + len(law))
    objs = bags(rng, np.asarray(EDGES * 2), d, law)
    cents = bags(rng, np.asarray([n, max(1, n - 1), n, max(1, n // 2)]), d, law)
    check(oracle_mod, objs, cents, run_all(d2, objs, cents), np.arange(objs.count))


@pytest.mark.parametrize("n", [16, 32, 64])
def test_bins(d2, oracle_mod, n):
    """A batch large enough to be sorted by size and cut into launches."""
    rng = np.random.default_rng(n)
    objs = bags(rng, rng.choice(EDGES, size=4500), 4, "far")
    cents = bags(rng, np.full(6, n), 4, "far")
    rows = np.sort(rng.choice(objs.count, size=120, replace=False))
    check(oracle_mod, objs, cents, run_all(d2, objs, cents), rows)


def run_pairs(d2, objs, cents, po, pc, precision, flows=True):
    import torch
    ctx = d2.Context(0, precision=precision)
    d2.d2_set_centroids(ctx, d2.bags_from_synth(cents, device="cuda:0"))
    ob = d2.bags_from_synth(objs, device="cuda:0")
    dist = torch.empty(len(po), dtype=torch.float64, device="cuda:0")
    st = torch.full((len(po),), 9, dtype=torch.int32, device="cuda:0")
    fl = (torch.empty((len(po), 127), dtype=torch.int32, device="cuda:0"),
          torch.empty((len(po), 127), dtype=torch.float64, device="cuda:0"))
    rc = d2.d2_mallows_batch(ctx, ob, torch.as_tensor(po, device="cuda:0"),
                             torch.as_tensor(pc, device="cuda:0"), dist,
                             flows=fl if flows else None, status=st)
    assert rc == d2.D2_OK
    d2.d2_sync(ctx)
    ctx.close()
    return dist.cpu().numpy(), st.cpu().numpy(), fl[0].cpu().numpy(), fl[1].cpu().numpy()


@pytest.mark.parametrize("law", ["normal", "lattice"])
@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("n,top", [(16, 16), (13, 48), (9, 64), (32, 16), (29, 32), (32, 64), (64, 64)])
def test_pair_lists(d2, oracle_mod, n, top, precision, law):
    """A list long enough for the lanes (24 pairs per SM of a 152-SM GPU), FP64
    throughout and FP32 with the FP64 test: values to FP64 optimality
    (2^-43 c_max plus rounding), plans that meet both marginals and cost D^2."""
    rng = np.random.default_rng(7 * n + top + precision)
    sizes = np.asarray([m for m in EDGES if m <= top] * 2)
    objs = bags(rng, sizes, 5, law)
    cents = bags(rng, np.full(4, n), 5, law)
    if precision == 1:
        objs = Bags(objs.loc.astype(np.float64), objs.w.astype(np.float64), objs.off, "f64", "f64")
        cents = Bags(cents.loc.astype(np.float64), cents.w.astype(np.float64), cents.off, "f64",
                     "f64")
    N, K = objs.count, cents.count
    t = 4096 + rng.integers(0, 9)
    po, pc = rng.integers(0, N, size=t), rng.integers(0, K, size=t)
    dist, st, cell, w = run_pairs(d2, objs, cents, po, pc, precision)
    assert (st == 0).all()
    _, _, ref = oracle_mod.assign(objs, cents, nthreads=8, return_all=True)
    ref = ref[po, pc]
    big = float(np.max(np.abs(objs.loc))) + float(np.max(np.abs(cents.loc)))
    floor = 1e-12 * objs.dim * big * big
    assert np.all(np.abs(dist - ref) <= 1e-11 * ref + floor)
    for q in rng.choice(t, size=60, replace=False):
        x, p = oracle_mod.bag(objs, int(po[q]))
        y, r = oracle_mod.bag(cents, int(pc[q]))
        ok = cell[q] >= 0
        assert ok.sum() == len(p) + len(r) - 1
        a, b, f = cell[q][ok] >> 16, cell[q][ok] & 0xFFFF, w[q][ok]
        assert (f >= 0).all()
        assert np.abs(np.bincount(a, weights=f, minlength=len(p)) - p / p.sum()).max() <= 1e-12
        assert np.abs(np.bincount(b, weights=f, minlength=len(r)) - r / r.sum()).max() <= 1e-12
        cost = float(np.dot(f, ((np.asarray(x)[a] - np.asarray(y)[b]) ** 2).sum(axis=1)))
        assert abs(cost - dist[q]) <= 1e-11 * dist[q] + floor


def test_pair_list_rejects_what_it_did(d2):
    """Bad indices and bad weights in a long list keep their status and error."""
    import torch
    rng = np.random.default_rng(5)
    objs = bags(rng, np.full(20, 8), 3, "normal")
    objs.w[objs.off[3]] = -1.0
    cents = bags(rng, np.full(4, 16), 3, "normal")
    po, pc = rng.integers(0, 20, size=5000), rng.integers(0, 4, size=5000)
    po[7], pc[9] = 20, -1
    ctx = d2.Context(0)
    d2.d2_set_centroids(ctx, d2.bags_from_synth(cents, device="cuda:0"))
    ob = d2.bags_from_synth(objs, device="cuda:0")
    dist = torch.empty(5000, dtype=torch.float64, device="cuda:0")
    st = torch.empty(5000, dtype=torch.int32, device="cuda:0")
    d2.d2_mallows_batch(ctx, ob, torch.as_tensor(po, device="cuda:0"),
                        torch.as_tensor(pc, device="cuda:0"), dist, status=st)
    with pytest.raises(d2.D2Error) as e:
        d2.d2_sync(ctx)
    assert e.value.code == d2.D2_EINVAL
    bad = (po == 20) | (pc == -1) | (po == 3)
    s, dd = st.cpu().numpy(), dist.cpu().numpy()
    assert (s[bad] == -1).all() and np.isnan(dd[bad]).all()
    assert (s[~bad] == 0).all() and np.isfinite(dd[~bad]).all()
    ctx.close()


def run_level(d2, objs, cents, iters, **kw):
    import torch
    ctx = d2.Context(0, **kw)
    d2.d2_set_centroids(ctx, d2.bags_from_synth(cents, device="cuda:0"))
    ob = d2.bags_from_synth(objs, device="cuda:0")
    loc = torch.empty(cents.loc.shape, dtype=torch.float64, device="cuda:0")
    w = torch.empty(cents.count, dtype=torch.float64, device="cuda:0")
    lab = torch.empty(objs.count, dtype=torch.int32, device="cuda:0")
    rc = d2.d2_cluster_level(ctx, ob, cents.count, objs.count, iters, loc, w, lab)
    assert rc == d2.D2_OK
    d2.d2_sync(ctx)
    ctx.close()
    return lab.cpu().numpy(), loc.cpu().numpy()


@pytest.mark.parametrize("kw", [{}, {"no_prune": True}, {"certify": 1}])
@pytest.mark.parametrize("N,lo,hi,n,K,law", [
    (300, 2, 48, 32, 6, "normal"),      # trees of more than 32 nodes, most pairs kept
    (300, 8, 16, 16, 6, "far"),         # few pairs kept: kept pairs without a saved basis
    (200, 16, 64, 64, 5, "normal"),
    (33000, 8, 16, 16, 64, "normal"),   # large enough that the kept share is counted
    (33000, 8, 16, 16, 64, "far"),
])
def test_level_agrees_with_the_warp_screen(d2, N, lo, hi, n, K, law, kw):
    """One segment of continuous bags: every LP has one optimal plan, so the
    labels are equal and the locations are the same sums; two FP32 units
    (2^-22) cover a stored location that rounds the other way.  A certified
    plan is only within 2^-24 of the optimal cost, so two cold starts may end
    in two of them: there the first round's labels are compared."""
    rng = np.random.default_rng(N + n)
    objs = bags(rng, rng.integers(lo, hi + 1, size=N), 6, law)
    cents = bags(rng, np.full(K, n), 6, law)
    for iters in (1,) if kw.get("certify") else (1, 4):
        a = run_level(d2, objs, cents, iters, **kw)
        b = run_level(d2, objs, cents, iters, start_rule=d2.D2_START_RANKED, **kw)
        assert np.array_equal(a[0], b[0])
        if kw.get("certify"):
            continue
        assert np.abs(a[1] - b[1]).max() <= 2.0 ** -22 * np.abs(b[1]).max()


@pytest.mark.parametrize("law", ["normal", "lattice"])
@pytest.mark.parametrize("n", [1, 16, 17, 32, 33, 64])
def test_assign_fp64_throughout(d2, oracle_mod, n, law):
    """FP64 assignments at the edges of their shapes, to FP64 optimality."""
    import torch
    rng = np.random.default_rng(31 * n + len(law))
    objs = bags(rng, np.asarray(EDGES * 2), 5, law)
    cents = bags(rng, np.asarray([n, max(1, n - 1), max(1, n // 2)]), 5, law)
    ctx = d2.Context(0, precision=1)
    d2.d2_set_centroids(ctx, d2.bags_from_synth(cents, device="cuda:0"))
    lab = torch.empty(objs.count, dtype=torch.int32, device="cuda:0")
    dist = torch.empty(objs.count, dtype=torch.float64, device="cuda:0")
    assert d2.d2_assign(ctx, d2.bags_from_synth(objs, device="cuda:0"), lab, dist) == d2.D2_OK
    d2.d2_sync(ctx)
    ctx.close()
    _, _, ref = oracle_mod.assign(objs, cents, nthreads=8, return_all=True)
    big = float(np.max(np.abs(objs.loc))) + float(np.max(np.abs(cents.loc)))
    floor = 1e-12 * objs.dim * big * big
    best = ref.min(axis=1)
    at = ref[np.arange(objs.count), lab.cpu().numpy()]
    assert np.all(at <= best * (1 + 1e-11) + floor)
    assert np.all(np.abs(dist.cpu().numpy() - at) <= 1e-11 * at + floor)
