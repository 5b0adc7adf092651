"""The window search by bounds with per-point weights against the search that
sums every window, and both kinds of weights at the sizes where the fold's
CTAs change.

The windows that are left are summed in the order of the tiled kernel, so
every output agrees bit for bit: for weights that hardly differ, differ by
orders of magnitude, or hold a few points that outweigh the rest, for residuals
without noise (exact ties) and without a dip.
"""

import numpy as np
import pytest

import paper_2607_00348_gb300 as pkg

from . import gpu_helpers as gh

pytestmark = pytest.mark.gpu

DY = ("near", "log", "heavy", "two", "tiny")


def _curve(n, days, flux, weights, seed):
    rng = np.random.default_rng(seed)
    t = np.sort(rng.uniform(0.0, days, n))
    dy = {"near": lambda: 1e-3 * rng.uniform(0.7, 1.3, n),
          "log": lambda: 1e-3 * np.exp(rng.normal(0.0, 1.5, n)),
          "heavy": lambda: np.where(np.arange(n) % 211 == 3, 1e-6, 1e-3),
          "two": lambda: np.where(t < 0.4 * days, 1e-3, 3e-3),
          "tiny": lambda: 1e-12 * rng.uniform(0.7, 1.3, n),
          "uniform": lambda: np.full(n, 1e-3)}[weights]()
    noise = rng.normal(0.0, 1.0, n) * np.minimum(dy, 1e-2)
    y = 1.0 + {"white": noise,
               "flat": np.zeros(n),
               "bright": np.abs(noise),
               "steps": -1e-3 * rng.integers(0, 2, n),
               "outliers": noise - 0.2 * (rng.random(n) < 0.002),
               "deep": noise - np.where((t - 0.3) % 2.9 < 0.11, 0.3, 0.0)}[flux]
    return t, y, dy


def _same(n, days, flux, weights, **kw):
    t, y, dy = _curve(n, days, flux, weights, n)
    got = []
    for flags in (4, 2):
        plan = pkg.Plan(pkg.PlanConfig(baseline_days=float(t[-1] - t[0]), n_points=n, test_flags=flags, **kw))
        got.append(gh.gpu_search(plan, t, y, dy))
        plan.close()
    (ra, a), (rb, b) = got
    for k in a:
        assert np.array_equal(a[k], b[k]), (k, np.flatnonzero(a[k] != b[k])[:5])
    assert ra.as_dict() == rb.as_dict()


@pytest.mark.parametrize("weights", DY)
@pytest.mark.parametrize("flux", ["white", "flat", "bright", "steps", "outliers", "deep"])
def test_weighted_bounds_keep_the_minimum(flux, weights):
    _same(3001, 40.0, flux, weights, period_min_days=0.7, period_max_days=12.0)


@pytest.mark.parametrize("weights", ["uniform", "near"])
@pytest.mark.parametrize("n", [31, 2048, 2049, 4096, 4097, 8192, 8193, 16385])
def test_bounds_where_the_fold_changes(n, weights):
    days = n * 0.0204 + 8.0
    _same(n, days, "white", weights, periods_days=np.geomspace(0.8, 0.5 * days, 40))


@pytest.mark.parametrize("n,days,kw", [
    (20011, 475.0, dict(periods_days=np.geomspace(0.5, 230.0, 300), k_min=41.39, k_max=546.94, q_cap=0.112)),
    (1440, 30.0, dict(period_min_days=0.6, period_max_days=14.0, dt0=0.2, refine_periods=40)),
    (62363, 1460.0, dict(periods_days=np.geomspace(0.5, 700.0, 60))),
    (100000, 2000.0, dict(periods_days=np.geomspace(0.5, 1000.0, 30), q_cap=0.05)),
    (144000, 3000.0, dict(periods_days=np.geomspace(0.5, 1500.0, 20))),
], ids=lambda v: str(v) if isinstance(v, int) else None)
@pytest.mark.parametrize("weights", ["near", "heavy"])
def test_weighted_bounds_over_sizes(n, days, kw, weights):
    _same(n, days, "white", weights, **kw)


def test_batch_of_both_kinds_equals_single_searches():
    import torch
    curves = [_curve(n, n * 0.03, "white", w, n) for n, w in ((1900, "near"), (4050, "uniform"), (9000, "log"), (3000, "two"))]
    cfgs = [pkg.PlanConfig(baseline_days=float(t[-1] - t[0]), n_points=t.size, period_min_days=0.8, period_max_days=14.0,
                           test_flags=4, refine_periods=10 * (i % 2)) for i, (t, _, _) in enumerate(curves)]
    plans = [pkg.Plan(c) for c in cfgs]
    alone = [gh.gpu_search(p, *c)[0].as_dict() for p, c in zip(plans, curves)]
    dev = torch.device("cuda:0")
    t, y, dy = (torch.as_tensor(np.concatenate([c[k] for c in curves]), device=dev) for k in range(3))
    batch = pkg.Batch(plans)
    offsets = np.cumsum([0] + [c[0].size for c in curves]).astype(np.int64)
    assert [r.as_dict() for r in batch.search(t, y, dy, offsets)] == alone
    batch.close()
    for p in plans:
        p.close()


@pytest.mark.parametrize("flux", ["steps", "flat", "deep"])
def test_periods_shared_by_several_ctas_of_the_tiled_kernel(flux):
    # at T0 step 1 a period has more than 2 x 65,536 windows, most of them equal
    _same(9001, 120.0, flux, "uniform", periods_days=np.geomspace(2.0, 50.0, 12), refine_periods=5)
