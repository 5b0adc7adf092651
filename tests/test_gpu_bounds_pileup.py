"""The window search by bounds after the fold through global memory: curves of
more points at a few phases than a super-bucket stages (every period here is
commensurate with the cadence or nearly so), for uniform and per-point weights,
bit for bit against the search that sums every window."""

import numpy as np
import pytest

import paper_2607_00348_gb300 as pkg

from . import gpu_helpers as gh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weights", ["uniform", "near", "heavy"])
@pytest.mark.parametrize("flux", ["white", "steps", "deep"])
@pytest.mark.parametrize("n", [9000, 20011])
def test_phase_pileup(n, flux, weights):
    rng = np.random.default_rng(n)
    t = 0.5 * np.arange(n)
    dy = {"uniform": np.full(n, 1e-3), "near": 1e-3 * rng.uniform(0.7, 1.3, n),
          "heavy": np.where(np.arange(n) % 211 == 3, 1e-6, 1e-3)}[weights]
    noise = rng.normal(0.0, 1.0, n) * dy
    y = 1.0 + {"white": noise, "steps": -1e-3 * rng.integers(0, 2, n),
               "deep": noise - np.where(t % 2.5 < 0.4, 0.01, 0.0)}[flux]
    periods = np.array([0.5, 0.75, 1.0, 1.0 + 1e-9, 1.25, 1.5, 2.0, 2.5, 3.0, 4.5, 7.0, 11.03, 20.0])
    got = []
    for flags in (0, 2):
        plan = pkg.Plan(pkg.PlanConfig(baseline_days=float(t[-1]), n_points=n, periods_days=periods, test_flags=flags))
        got.append(gh.gpu_search(plan, t, y, dy))
        plan.close()
    (ra, a), (rb, b) = got
    for k in a:
        assert np.array_equal(a[k], b[k]), (k, np.flatnonzero(a[k] != b[k])[:5])
    assert ra.as_dict() == rb.as_dict()
