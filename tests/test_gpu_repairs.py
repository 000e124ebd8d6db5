"""Bags of nearly coinciding supports: the FP32 basis is far from the FP64
optimum in pivots, so most pairs leave the lanes for the warp-per-pair kernels."""
import numpy as np
import pytest

from test_gpu_lanes import check, d2, run_all, run_pairs  # noqa: F401  (d2: the fixture)

from paper_1302_0435_gb300.synth import Bags

pytestmark = pytest.mark.gpu


def near(rng, count, n, d, points):
    """Bags of n supports of equal weight, each within 1e-4 of one of a few points."""
    loc = points[rng.integers(0, len(points), size=count * n)] + 1e-4 * rng.normal(size=(count * n, d))
    return Bags(loc.astype(np.float32), np.full(count * n, 1.0 / n, np.float32),
                np.arange(count + 1, dtype=np.int64) * n, "f32", "f32")


@pytest.mark.parametrize("m,n", [(16, 16), (12, 16), (32, 32), (40, 16), (64, 64)])
def test_nearly_coinciding_supports(d2, oracle_mod, m, n):  # noqa: F811
    rng = np.random.default_rng(m + n)
    points = rng.normal(size=(3, 6))
    objs, cents = near(rng, 40, m, 6, points), near(rng, 5, n, 6, points)
    check(oracle_mod, objs, cents, run_all(d2, objs, cents), np.arange(objs.count))
    t = 4001
    po, pc = rng.integers(0, objs.count, size=t), rng.integers(0, cents.count, size=t)
    dist, st, cell, w = run_pairs(d2, objs, cents, po, pc, 0)
    assert (st == 0).all()
    _, _, ref = oracle_mod.assign(objs, cents, nthreads=8, return_all=True)
    big = float(np.max(np.abs(objs.loc))) + float(np.max(np.abs(cents.loc)))
    assert np.all(np.abs(dist - ref[po, pc]) <= 1e-11 * ref[po, pc] + 1e-12 * 6 * big * big)
    for q in rng.choice(t, size=40, replace=False):
        ok = cell[q] >= 0
        a, b, f = cell[q][ok] >> 16, cell[q][ok] & 0xFFFF, w[q][ok]
        assert ok.sum() == m + n - 1 and (f >= 0).all()
        assert np.abs(np.bincount(a, weights=f, minlength=m) - 1 / m).max() <= 1e-12
        assert np.abs(np.bincount(b, weights=f, minlength=n) - 1 / n).max() <= 1e-12
