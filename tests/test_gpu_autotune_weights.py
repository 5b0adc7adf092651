"""The autotuner's probe runs what the search runs: its waves leave the chi2,
duration, start and depth of the periods they cover (here all of them) as the
search does, for curves with one uncertainty and with their own."""

import numpy as np
import pytest

import paper_2607_00348_gb300 as pkg

from . import gpu_helpers as gh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own", [(True,), (False, True), (True, False, True)])
def test_probe_of_curves_with_own_uncertainties(own):
    import torch
    rng = np.random.default_rng(len(own))
    sizes = [1900 + 1150 * i for i in range(len(own))]
    t = [np.sort(rng.uniform(0.0, 30.0, n)) for n in sizes]
    dy = [1e-3 * (rng.uniform(0.7, 1.3, n) if o else np.ones(n)) for n, o in zip(sizes, own)]
    y = [1.0 + rng.normal(0.0, 1e-3, n) for n in sizes]
    plans = [pkg.Plan(pkg.PlanConfig(baseline_days=30.0, n_points=n, periods_days=np.geomspace(0.9, 14.0, 150 + 7 * i)))
             for i, n in enumerate(sizes)]
    dev = torch.device("cuda:0")
    args = [torch.as_tensor(np.concatenate(a), device=dev) for a in (t, y, dy)]
    args.append(np.cumsum([0] + sizes).astype(np.int64))
    batch = pkg.Batch(plans)
    batch.autotune(*args)
    probed = [gh.batch_outputs(batch, i, p.n_periods) for i, p in enumerate(plans)]
    batch.search(*args)
    for i, p in enumerate(plans):
        searched = gh.batch_outputs(batch, i, p.n_periods)
        for k in ("chi2", "dur_idx", "t0_idx", "depth", "t0"):
            assert np.array_equal(probed[i][k], searched[k]), (i, k)
    batch.close()
    for p in plans:
        p.close()
