"""Bags that no pair can be solved for, beside ordinary ones: the ordinary
bags' results are those of a call without the others."""
import contextlib

import numpy as np
import pytest

from paper_1302_0435_gb300.synth import Bags

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def d2():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_0435_gb300 import build, d2 as mod
    build.build()
    mod.load()
    return mod


def bags(rng, sizes, d, spread=0.0):
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    T = int(off[-1])
    loc = rng.normal(size=(T, d)) + np.repeat(rng.normal(0, spread, size=(len(sizes), d)), sizes,
                                              axis=0)
    return Bags(loc.astype(np.float32), rng.exponential(size=T).astype(np.float32), off, "f32",
                "f32")


def spoil(objs, rows, kind):
    """The bags of `rows` given locations whose costs are not finite in FP32."""
    loc = objs.loc.copy()
    for i in rows:
        s = slice(objs.off[i], objs.off[i + 1])
        if kind == "nan":
            loc[objs.off[i], 0] = np.nan
        elif kind == "inf":
            loc[s, 1] = np.inf
        else:  # finite, but their squares overflow
            loc[s] *= np.float32(1e25)
    return Bags(loc, objs.w, objs.off, "f32", "f32")


@pytest.mark.parametrize("rule", [0, 1])  # lanes, and a warp per pair
@pytest.mark.parametrize("n,top", [(16, 16), (12, 8), (13, 12), (16, 24)])
@pytest.mark.parametrize("kind", ["nan", "inf", "overflow"])
def test_level_beside_non_finite_bags(d2, kind, n, top, rule):
    """The first round of a level starts small trees from the supports' order
    along a direction of the object, which such bags do not have.  The sums of
    a round run over the members in order, so the other bags' labels and the
    locations are the same bits as without them."""
    import torch
    rng = np.random.default_rng(n + top)
    N, K = 400, 6
    objs = bags(rng, rng.integers(max(1, top // 2), top + 1, size=N), 6, 2.0)
    cents = bags(rng, np.full(K, n), 6, 2.0)
    rows = np.arange(N) % 9 == 4
    out = []
    for o in (objs.subset(np.flatnonzero(~rows)), spoil(objs, np.flatnonzero(rows), kind)):
        ctx = d2.Context(0, start_rule=rule)
        d2.d2_set_centroids(ctx, d2.bags_from_synth(cents, device="cuda:0"))
        loc = torch.empty(cents.loc.shape, dtype=torch.float64, device="cuda:0")
        w = torch.empty(K, dtype=torch.float64, device="cuda:0")
        lab = torch.empty(o.count, dtype=torch.int32, device="cuda:0")
        d2.d2_cluster_level(ctx, d2.bags_from_synth(o, device="cuda:0"), K, o.count, 4, loc, w, lab)
        d2.d2_sync(ctx)
        ctx.close()
        out.append((lab.cpu().numpy(), loc.cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0][~rows])
    assert np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("kind", ["nan", "inf", "overflow"])
def test_pairs_beside_non_finite_bags(d2, kind):
    """A short list, a warp per pair from the ranked staircase."""
    import torch
    rng = np.random.default_rng(3)
    objs = bags(rng, rng.integers(2, 17, size=60), 6)
    cents = bags(rng, np.full(5, 16), 6)
    rows = np.arange(60) % 7 == 3
    po, pc = rng.integers(0, 60, size=500), rng.integers(0, 5, size=500)
    out = []
    for o in (objs, spoil(objs, np.flatnonzero(rows), kind)):
        ctx = d2.Context(0)
        d2.d2_set_centroids(ctx, d2.bags_from_synth(cents, device="cuda:0"))
        dist = torch.empty(500, dtype=torch.float64, device="cuda:0")
        d2.d2_mallows_batch(ctx, d2.bags_from_synth(o, device="cuda:0"),
                            torch.as_tensor(po, device="cuda:0"),
                            torch.as_tensor(pc, device="cuda:0"), dist)
        with contextlib.suppress(d2.D2Error):  # those bags' own pairs
            d2.d2_sync(ctx)
        ctx.close()
        out.append(dist.cpu().numpy())
    keep = ~rows[po]
    assert np.array_equal(out[0][keep], out[1][keep])


def rejected(N, top, n, K, seed):
    """N bags of up to `top` supports, one without a support and one above the
    bound, and their indices."""
    rng = np.random.default_rng(seed)
    sizes = rng.integers(max(1, top // 2), top + 1, size=N)
    bad = np.asarray([N // 3, 2 * N // 3])
    sizes[bad] = 0, top + 1
    return bags(rng, sizes, 6, 2.0), bags(rng, np.full(K, n), 6, 2.0), bad


# bags, bound, supports of a centroid: one launch; cut by size, with the bad
# bags in no launch
REJECT = [(600, 16, 16), (5000, 12, 18), (5000, 64, 40), ((1 << 17) + 1, 16, 16)]


@pytest.mark.parametrize("rule", [0, 1])
@pytest.mark.parametrize("N,top,n", REJECT)
def test_rejected_bags_have_no_result(d2, N, top, n, rule):
    """Label -1, NaN distances and D2_EINVAL, whatever the buffers held; the
    other bags as without them."""
    import torch
    objs, cents, bad = rejected(N, top, n, 8, N + n)
    ok = np.ones(N, bool)
    ok[bad] = False
    out = []
    for o in (objs, objs.subset(np.flatnonzero(ok))):
        ob = d2.bags_from_synth(o, device="cuda:0")
        ob.s.max_support = top
        ctx = d2.Context(0, start_rule=rule)
        d2.d2_set_centroids(ctx, d2.bags_from_synth(cents, device="cuda:0"))
        lab = torch.full((o.count,), 5, dtype=torch.int32, device="cuda:0")
        dist = torch.full((o.count,), 5.0, dtype=torch.float64, device="cuda:0")
        lab2, dist2 = lab.clone(), dist.clone()
        every = torch.full((o.count, 8), 5.0, dtype=torch.float64, device="cuda:0")
        eps = torch.zeros(1, dtype=torch.float64, device="cuda:0")
        for call in (lambda: d2.d2_assign(ctx, ob, lab, dist, eps=eps),
                     lambda: d2.d2_mallows_all(ctx, ob, every, lab2, dist2)):
            call()
            if o is objs:
                with pytest.raises(d2.D2Error) as e:
                    d2.d2_sync(ctx)
                assert e.value.code == d2.D2_EINVAL
            else:
                d2.d2_sync(ctx)
        ctx.close()
        out.append([t.cpu().numpy() for t in (lab, dist, lab2, dist2, every, eps)])
    lab, dist, lab2, dist2, every, eps = out[0]
    assert (lab[bad] == -1).all() and (lab2[bad] == -1).all()
    assert np.isnan(dist[bad]).all() and np.isnan(dist2[bad]).all() and np.isnan(every[bad]).all()
    assert np.isnan(eps[0])
    for a, b in zip(out[0][:5], out[1][:5]):
        assert np.array_equal(a[ok], b)


@pytest.mark.parametrize("N,top,n", REJECT)
def test_rejected_bags_in_a_level(d2, N, top, n):
    """Two levels: the bags without a label stay without one, and the others'
    labels are those of the merged centroids."""
    import torch
    K = 8
    objs, cents, bad = rejected(N, top, n, K, N + n)
    ob = d2.bags_from_synth(objs, device="cuda:0")
    ob.s.max_support = top
    ctx = d2.Context(0)
    d2.d2_set_centroids(ctx, d2.bags_from_synth(cents, device="cuda:0"))
    loc = torch.empty(cents.loc.shape, dtype=torch.float64, device="cuda:0")
    w = torch.empty(K, dtype=torch.float64, device="cuda:0")
    lab = torch.full((N,), 5, dtype=torch.int32, device="cuda:0")
    with pytest.raises(d2.D2Error) as e:
        d2.d2_cluster_level(ctx, ob, K, N // 3, 3, loc, w, lab)
    assert e.value.code == d2.D2_EINVAL
    lab = lab.cpu().numpy()
    assert (lab[bad] == -1).all()
    ok = np.ones(N, bool)
    ok[bad] = False
    assert (lab[ok] >= 0).all() and (lab[ok] < K).all()
    assert w.cpu().numpy().sum() == N - 2
    ctx.close()
