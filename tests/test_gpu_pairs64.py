"""Long pair lists in FP64 throughout: small trees come to the lanes from 64
pairs per SM, and pairs are priced by the lanes' candidates of the last scan."""
import numpy as np
import pytest

from test_gpu_lanes import EDGES, bags, d2, run_pairs  # noqa: F401  (d2: the fixture)

from paper_1302_0435_gb300.synth import Bags

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("law", ["normal", "lattice"])
@pytest.mark.parametrize("n,top", [(16, 16), (3, 12), (16, 48), (16, 64), (20, 8), (32, 32),
                                   (17, 33), (32, 64), (33, 9), (64, 64)])
def test_long_lists_in_fp64(d2, oracle_mod, n, top, law):  # noqa: F811
    """Values to FP64 optimality (2^-43 c_max plus rounding), plans that meet
    both marginals and cost D^2."""
    rng = np.random.default_rng(100 * n + top)
    f64 = lambda b: Bags(b.loc.astype(np.float64), b.w.astype(np.float64), b.off, "f64", "f64")
    objs = f64(bags(rng, np.asarray([m for m in EDGES if m <= top] * 2), 5, law))
    cents = f64(bags(rng, np.asarray([n, n, max(1, n - 1), max(1, n // 2)]), 5, law))
    t = 10007
    po, pc = rng.integers(0, objs.count, size=t), rng.integers(0, cents.count, size=t)
    dist, st, cell, w = run_pairs(d2, objs, cents, po, pc, 1)
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
