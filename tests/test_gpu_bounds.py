"""The bounds kernel of the window search against the search that sums every
window (test_flags bits 2 and 1): the same minimum, duration, start and bits of chi2
at every period.

Ruling a window out never changes the minimum, and the windows that are left
are summed in the order of the tiled kernel, so the two searches agree bit
for bit whatever the data: white noise, constant and zero residuals (signed
zeros decide), strong trends, outliers, one deep transit, tiny and huge
residuals, and curves with one or several staged tiles.
"""

import numpy as np
import pytest

import paper_2607_00348_gb300 as pkg

from . import gpu_helpers as gh

pytestmark = pytest.mark.gpu


def _flux(kind, t, rng):
    n = t.size
    noise = rng.normal(0.0, 1e-3, n)
    if kind == "white":
        return 1.0 + noise
    if kind == "flat":
        return np.ones(n)
    if kind == "bright":            # no window has a positive depth
        return 1.0 + np.abs(noise)
    if kind == "offset":            # every window has one
        return 0.9 + noise
    if kind == "steps":             # many exactly equal windows
        return 1.0 - 1e-3 * (rng.integers(0, 2, n))
    if kind == "trend":
        return 1.0 + noise + 0.05 * np.sin(2.0 * np.pi * t / 11.3) + 1e-3 * t
    if kind == "outliers":
        noise[rng.integers(0, n, 5)] -= 0.2
        noise[rng.integers(0, n, 5)] += 0.5
        return 1.0 + noise
    if kind == "deep":
        return 1.0 + noise - np.where((t - 0.3) % 2.9 < 0.11, 0.3, 0.0)
    if kind == "tiny":
        return 1.0 + 1e-9 * noise
    return 1.0 + 1e4 * noise        # huge


def _both(n, days, flux, **kw):
    rng = np.random.default_rng(n)
    t = np.sort(rng.uniform(0.0, days, n))
    y = _flux(flux, t, rng)
    dy = np.full(n, 1e-3)
    got = []
    for flags in (4, 2):
        plan = pkg.Plan(pkg.PlanConfig(baseline_days=float(t[-1] - t[0]), n_points=n, test_flags=flags, **kw))
        got.append(gh.gpu_search(plan, t, y, dy))
        plan.close()
    (ra, a), (rb, b) = got
    for k in a:
        assert np.array_equal(a[k], b[k]), (k, np.flatnonzero(a[k] != b[k])[:5])
    assert ra.as_dict() == rb.as_dict()


@pytest.mark.parametrize("flux", ["white", "flat", "bright", "offset", "steps", "trend", "outliers", "deep", "tiny", "huge"])
def test_bounds_rule_out_only_windows_above_the_minimum(flux):
    _both(3001, 40.0, flux, period_min_days=0.7, period_max_days=12.0)


@pytest.mark.parametrize("n,days,kw", [
    (24, 9.0, dict(periods_days=np.geomspace(0.9, 4.0, 23))),
    (511, 20.0, dict(period_min_days=0.6, period_max_days=9.0, dt0=0.2)),
    (1440, 30.0, dict(period_min_days=0.6, period_max_days=14.0, refine_periods=60)),
    (2500, 30.0, dict(period_min_days=0.6, period_max_days=14.0, k_min=41.39, k_max=546.94, q_cap=0.112, dt0=0.01)),
    (20480, 300.0, dict(periods_days=np.geomspace(0.5, 140.0, 300))),
    (62363, 1460.0, dict(periods_days=np.geomspace(0.5, 700.0, 311))),
    (62363, 1460.0, dict(periods_days=np.geomspace(0.5, 700.0, 40), u1=0.9, u2=0.05, refine_periods=5)),
    (144000, 3000.0, dict(periods_days=np.geomspace(0.5, 1500.0, 97))),
    (260000, 3000.0, dict(periods_days=np.geomspace(0.5, 1500.0, 13))),
], ids=lambda v: str(v) if isinstance(v, int) else None)
def test_bounds_over_sizes_and_options(n, days, kw):
    _both(n, days, "white", **kw)
