"""The window search by bounds where delta-chi2 leaves the normal range of
FP32: uniform uncertainties so large that its values are subnormal (so coarse
that many windows are equal, and the first one decides) or vanish, or so small
that they overflow.  Equal, bit for bit, to the search that sums every window.
"""

import numpy as np
import pytest

import paper_2607_00348_gb300 as pkg

from . import gpu_helpers as gh

pytestmark = pytest.mark.gpu


def _same(n, y, dy, **kw):
    rng = np.random.default_rng(n)
    t = np.sort(rng.uniform(0.0, 40.0, n))
    got = []
    for flags in (0, 2):
        plan = pkg.Plan(pkg.PlanConfig(baseline_days=40.0, n_points=n, test_flags=flags, **kw))
        got.append(gh.gpu_search(plan, t, y, dy)[1])
        plan.close()
    a, b = got
    for k in a:
        assert np.array_equal(a[k], b[k], equal_nan=True), (k, np.flatnonzero(a[k] != b[k])[:5])


@pytest.mark.parametrize("n", [700, 3001, 9001])
@pytest.mark.parametrize("dy", [1e14, 1e16, 1e17, 1e18, 3e18, 1e19, 3e19, 1e20, 1e21, 1e-17, 1e-19, 1e-20])
def test_uniform_uncertainty_of_any_size(n, dy):
    y = 1.0 + np.random.default_rng(n + 1).normal(0.0, 1e-3, n)
    _same(n, y, np.full(n, dy), period_min_days=0.7, period_max_days=12.0)


@pytest.mark.parametrize("dy", [1e6, 1e8, 1e10, 1e11, 1e12, 1e13])
def test_own_uncertainties_of_any_size(dy):
    rng = np.random.default_rng(3)
    y = 1.0 + rng.normal(0.0, 1e-9, 3001)
    _same(3001, y, dy * rng.uniform(0.7, 1.3, 3001), period_min_days=0.7, period_max_days=12.0)
