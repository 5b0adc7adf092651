"""More than 64 durations at a period: refused by every search of the tiled
plan, whatever the curve and whether its windows would be ruled out or not."""

import numpy as np
import pytest

import paper_2607_00348_gb300 as pkg

from . import gpu_helpers as gh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, 2])
@pytest.mark.parametrize("n,ratio", [(3001, 1.02), (160001, 1.02), (160001, 1.05)])   # the last: 64 but for those too long for a tile
def test_more_durations_than_a_period_may_have(n, ratio, flags):
    rng = np.random.default_rng(1)
    t = np.sort(rng.uniform(0.0, 400.0, n))
    plan = pkg.Plan(pkg.PlanConfig(baseline_days=400.0, n_points=n, periods_days=np.array([28.5, 30.6]), dt0=1.0,
                                   dur_ratio=ratio, test_flags=flags))
    with pytest.raises(pkg.GtlsError, match="check 19"):
        gh.gpu_search(plan, t, 1.0 + rng.normal(0.0, 1e-3, n), np.full(n, 1e-3))
    plan.close()
