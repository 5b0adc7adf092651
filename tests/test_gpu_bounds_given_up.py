"""Curves whose windows the bounds cannot tell apart: outliers above the flux,
a flux far from 1, no dip at all, and curves that change from one to another.
Periods are given up in the walk, at the list or untried, and all outputs are
bit for bit those of the search that sums every window, in one wave, in several
and in a batch with a well-behaved curve."""

import numpy as np
import pytest

import paper_2607_00348_gb300 as pkg

from . import gpu_helpers as gh

pytestmark = pytest.mark.gpu


def _curve(n, kind, own_dy):
    rng = np.random.default_rng(n)
    t = np.sort(rng.uniform(0.0, 60.0, n))
    noise = rng.normal(0.0, 1e-4, n)
    spike = 0.5 * (rng.random(n) < 0.004)
    y = {"white": 1.0 + noise, "above": 1.0 + noise + spike, "low": 0.9 + noise, "bright": 1.0 + np.abs(noise),
         "half": 1.0 + noise + spike * (t > 30.0)}[kind]
    return t, y, 1e-4 * rng.uniform(0.8, 1.2, n) if own_dy else np.full(n, 1e-4)


def _plan(n, flags, **kw):
    return pkg.Plan(pkg.PlanConfig(baseline_days=60.0, n_points=n, test_flags=flags,
                                   periods_days=np.geomspace(0.6, 29.0, 300), **kw))


def _equal(a, b):
    for k in a:
        assert np.array_equal(a[k], b[k]), (k, np.flatnonzero(a[k] != b[k])[:5])


@pytest.mark.parametrize("own_dy", [False, True])
@pytest.mark.parametrize("kind", ["above", "low", "bright", "half"])
@pytest.mark.parametrize("n", [1440, 4001, 9001, 30011])
def test_given_up_periods(n, kind, own_dy):
    c = _curve(n, kind, own_dy)
    every = _plan(n, 2, refine_periods=0 if own_dy else 40)
    ra, a = gh.gpu_search(every, *c)
    every.close()
    for chunk in (0, 70):
        some = _plan(n, 0, periods_per_chunk=chunk, refine_periods=0 if own_dy else 40)
        rb, b = gh.gpu_search(some, *c)
        some.close()
        _equal(b, a)
        assert ra.as_dict() == rb.as_dict()


def test_batch_of_curves_given_up_and_not():
    import torch
    dev = torch.device("cuda:0")
    shapes = [(4001, "white", False), (3801, "above", False), (4010, "low", False), (3900, "above", True), (4001, "white", True)]
    curves = [_curve(*s) for s in shapes]
    plans = [_plan(s[0], 0) for s in shapes]
    batch = pkg.Batch(plans, wave_slots=200)
    for _ in range(2):
        batch.search(*(torch.as_tensor(np.concatenate([c[k] for c in curves]), device=dev) for k in range(3)),
                     np.cumsum([0] + [s[0] for s in shapes]).astype(np.int64))
        for i, (s, c) in enumerate(zip(shapes, curves)):
            every = _plan(s[0], 2)
            _equal(gh.batch_outputs(batch, i, 300), gh.gpu_search(every, *c)[1])
            every.close()
    batch.close()
    for p in plans:
        p.close()
