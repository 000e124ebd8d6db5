"""Which screen a level's rounds run, and each of them against the others and
the oracle."""
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


def run_level(d2, objs, cents, iters, seg=None, **kw):
    """Labels, locations and the change of the library's counters."""
    import torch
    ctx = d2.Context(0, **kw)
    d2.d2_set_centroids(ctx, d2.bags_from_synth(cents, device="cuda:0"))
    ob = d2.bags_from_synth(objs, device="cuda:0")
    loc = torch.empty(cents.loc.shape, dtype=torch.float64, device="cuda:0")
    w = torch.empty(cents.count, dtype=torch.float64, device="cuda:0")
    lab = torch.empty(objs.count, dtype=torch.int32, device="cuda:0")
    s0 = d2.d2_get_stats()
    d2.d2_cluster_level(ctx, ob, cents.count, seg or objs.count, iters, loc, w, lab)
    d2.d2_sync(ctx)
    s1 = d2.d2_get_stats()
    ctx.close()
    return lab.cpu().numpy(), loc.cpu().numpy(), {k: s1[k] - s0[k] for k in s1}


@pytest.mark.parametrize("kw", [{"no_prune": True}, {"certify": 1}])
@pytest.mark.parametrize("tuned", [False, True])
@pytest.mark.parametrize("n,top", [(32, 48), (16, 64)])
def test_level_of_full_bases_runs_as_the_warp_screen(d2, n, top, tuned, kw):
    """An unpruned level that keeps full bases solves a warp per pair: the same
    launches (cuts by tree size, and where nothing fixes the launch shape its
    timing) and the same bits as with the cold start fixed."""
    rng = np.random.default_rng(n + top)
    objs = bags(rng, rng.integers(2, top + 1, size=9000), 5, 1.0)
    cents = bags(rng, np.full(6, n), 5, 1.0)
    kw = dict(kw, group_lanes=0 if tuned else 32)
    a = run_level(d2, objs, cents, 4, **kw)
    b = run_level(d2, objs, cents, 4, start_rule=d2.D2_START_RANKED, **kw)
    assert a[2]["kernel_launches"] == b[2]["kernel_launches"]
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


def test_level_of_full_bases_is_tuned(d2):
    """Its bins of 8,192 objects and more are timed on the first round; two
    starts of continuous bags end in the one optimal plan (the labels are
    equal, the locations differ by FP32 units)."""
    rng = np.random.default_rng(8)
    objs = bags(rng, rng.integers(2, 49, size=20000), 5, 1.0)
    cents = bags(rng, np.full(6, 32), 5, 1.0)
    a = run_level(d2, objs, cents, 3, no_prune=True)
    b = run_level(d2, objs, cents, 3, no_prune=True, group_lanes=32)
    assert a[2]["kernel_launches"] > b[2]["kernel_launches"]
    assert np.array_equal(a[0], b[0])
    assert np.abs(a[1] - b[1]).max() <= 2.0 ** -22 * np.abs(b[1]).max()


@pytest.mark.parametrize("n,top", [(16, 16), (8, 24)])
def test_small_level_of_small_trees_runs_as_the_warp_screen(d2, n, top):
    """Trees of at most 32 nodes, few objects: the launches and bits of a level
    with its cold start fixed."""
    rng = np.random.default_rng(n)
    objs = bags(rng, rng.integers(2, top + 1, size=700), 6, 3.0)
    cents = bags(rng, np.full(10, n), 6, 3.0)
    a = run_level(d2, objs, cents, 5)
    b = run_level(d2, objs, cents, 5, start_rule=d2.D2_START_RANKED)
    assert a[2]["kernel_launches"] == b[2]["kernel_launches"]
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("N,seg,n,lo,top", [
    (900, 900, 16, 2, 40),     # lane rounds, the exact pass by warps for want of bags
    (1500, 1500, 16, 2, 40),   # lane rounds and exact pass, trees above 32 nodes
    (7000, 7000, 16, 8, 16),   # lane rounds and exact pass
    (2000, 500, 32, 2, 40),    # and a merged level, its exact pass by warps
    (600, 200, 64, 16, 64),    # a merged level by lanes throughout
])
def test_level_routes_agree(d2, N, seg, n, lo, top):
    """Continuous bags have one optimal plan: the routes' labels are equal and
    the locations differ by FP32 units."""
    rng = np.random.default_rng(N + n)
    objs = bags(rng, rng.integers(lo, top + 1, size=N), 6, 3.0)
    cents = bags(rng, np.full(8, n), 6, 3.0)
    a = run_level(d2, objs, cents, 4, seg)
    b = run_level(d2, objs, cents, 4, seg, start_rule=d2.D2_START_RANKED)
    assert np.array_equal(a[0], b[0])
    assert np.abs(a[1] - b[1]).max() <= 2.0 ** -22 * np.abs(b[1]).max()


# 1 MiB holds a byte a tree node of every pair, not the 3 or 11 of the other
# stores: the rounds run by lanes, warm, where the level is not pruned.
# (N, K, most supports, supports of a centroid): N * K * (top + n) bytes
WARM_LANES = [
    (1200, 24, 16, 16),   # 32 nodes, from the staircase, exact pass by lanes
    (400, 40, 32, 16),    # the other shapes start row by row; exact pass by warps
    (400, 40, 16, 30),
    (1100, 14, 24, 32),
    (600, 16, 64, 32),
    (300, 20, 64, 64),    # exact pass by lanes
    (300, 20, 32, 60),
]


@pytest.mark.parametrize("kw", [{"no_prune": True}, {"certify": 1}])
@pytest.mark.parametrize("N,K,top,n", WARM_LANES)
def test_warm_rounds_of_all_pairs_by_lanes(d2, oracle_mod, N, K, top, n, kw):
    """Every round's labels are nearest centroids of the locations the round
    before left (read from a run of one round less), by the oracle."""
    assert 3 * N * K * (top + n) > 2 ** 20 >= N * K * (top + n)
    rng = np.random.default_rng(N + top + n)
    sizes = rng.integers(max(1, top // 4), top + 1, size=N)
    sizes[:3] = top, 1, top
    objs = bags(rng, sizes, 5, 1.0)
    cents = bags(rng, np.full(K, n), 5, 1.0)
    cents = Bags(cents.loc, np.full(K * n, 1.0 / n, np.float32), cents.off, "f32", "f32")
    runs = [run_level(d2, objs, cents, t, warm_budget_mib=1, **kw) for t in (2, 3, 4)]
    whole = run_level(d2, objs, cents, 4, **kw)  # room for full bases: a warp per pair
    # another screen: other launches, or other pivots from another start
    screen = lambda r: (r[2]["kernel_launches"], r[2]["pivots_screened"])
    assert screen(whole) != screen(runs[2])
    for s in (whole[2], runs[2][2]):
        assert s["pairs_screened"] == 4 * N * K
        if kw.get("certify"):
            assert s["pairs_certified"] >= 0.99 * 4 * N * K
    for before, after in ((runs[0], runs[1]), (runs[1], runs[2])):
        at = Bags(before[1].astype(np.float32), cents.w, cents.off, "f32", "f32")
        _, _, ref = oracle_mod.assign(objs, at, nthreads=8, return_all=True)
        got = ref[np.arange(N), after[0]]
        assert np.all(got <= ref.min(axis=1) * (1 + 1e-7) + 1e-9)


def test_pruned_rounds_by_lanes_with_little_memory(d2):
    """Where only the byte store fits, and where none does, a pruned level has
    the labels and locations of one with room."""
    rng = np.random.default_rng(77)
    objs = bags(rng, rng.integers(2, 33, size=1500), 5, 4.0)
    cents = bags(rng, np.full(12, 30), 5, 4.0)  # 62 nodes: 1.1 MB of bytes
    out = [run_level(d2, objs, cents, 4, warm_budget_mib=b) for b in (0, 2, 1)]
    for o in out[1:]:
        assert np.array_equal(o[0], out[0][0])
        assert np.abs(o[1] - out[0][1]).max() <= 2.0 ** -22 * np.abs(out[0][1]).max()
