"""Waves of the window search by bounds: what one wave lists (windows to sum
again, periods for the tiled kernel) is its own.

Every wave starts with empty lists, whatever the wave, the search or the batch
loop before it left there, so that a search in many small waves, searches of
unlike curves one after the other with one plan, and batches of several loops
all equal the search that sums every window (test_flags 2) bit for bit.
"""

import numpy as np
import pytest

import paper_2607_00348_gb300 as pkg

from . import gpu_helpers as gh

pytestmark = pytest.mark.gpu

KINDS = ("white", "flat", "steps")   # few windows listed; every period left to the tiled kernel; many windows listed


def _curve(n, kind, own_dy, seed):
    rng = np.random.default_rng(seed)
    t = np.sort(rng.uniform(0.0, 20.0, n))
    y = {"white": lambda: 1.0 + rng.normal(0.0, 1e-3, n),
         "flat": lambda: np.ones(n),
         "steps": lambda: 1.0 - 1e-3 * rng.integers(0, 2, n)}[kind]()
    return t, y, 1e-3 * rng.uniform(0.7, 1.3, n) if own_dy else np.full(n, 1e-3)


def _plan(n, flags, **kw):
    return pkg.Plan(pkg.PlanConfig(baseline_days=20.0, n_points=n, test_flags=flags, **kw))


def _equal(a, b):
    for k in a:
        assert np.array_equal(a[k], b[k]), (k, np.flatnonzero(a[k] != b[k])[:5])


@pytest.mark.parametrize("own_dy", [False, True])
@pytest.mark.parametrize("n,chunk", [(24, 1), (31, 7), (400, 3), (3001, 50)])
def test_small_waves_of_unlike_curves(n, chunk, own_dy):
    kw = dict(periods_days=np.geomspace(0.9, 9.0, 101), refine_periods=0 if own_dy else 9)
    every = _plan(n, 2, **kw)
    some = _plan(n, 0, periods_per_chunk=chunk, **kw)
    for i, kind in enumerate(KINDS + KINDS[::-1]):
        c = _curve(n, kind, own_dy, 100 * n + i)
        rb, b = gh.gpu_search(every, *c)
        ra, a = gh.gpu_search(some, *c)
        _equal(a, b)
        assert ra.as_dict() == rb.as_dict()
    # one kernel more per wave: the bounds are on in the one plan only
    waves = -(-101 // chunk) + (-(-9 // chunk) if not own_dy else 0)
    assert some.profile().window_search_launches == waves
    assert some.profile().kernel_launches == every.profile().kernel_launches + 4 * waves - 3 * (1 if own_dy else 2)
    every.close()
    some.close()


def test_batch_loops_in_small_waves():
    import torch
    dev = torch.device("cuda:0")
    shapes = [(n, kind, own) for n in (24, 1900, 4050) for kind in KINDS for own in (False, True)]
    curves = [_curve(n, kind, own, i) for i, (n, kind, own) in enumerate(shapes)]
    kw = [dict(periods_days=np.geomspace(0.9, 9.0, 37 + 5 * i), refine_periods=4 * (i % 2)) for i in range(len(shapes))]
    plans = [_plan(s[0], 0, **k) for s, k in zip(shapes, kw)]
    t, y, dy = (torch.as_tensor(np.concatenate([c[k] for c in curves]), device=dev) for k in range(3))
    offsets = np.cumsum([0] + [s[0] for s in shapes]).astype(np.int64)
    batch = pkg.Batch(plans, wave_slots=11)
    for _ in range(2):
        batch.search(t, y, dy, offsets)
        for i, (s, c) in enumerate(zip(shapes, curves)):
            every = _plan(s[0], 2, **kw[i])
            _, b = gh.gpu_search(every, *c)
            every.close()
            _equal(gh.batch_outputs(batch, i, plans[i].n_periods), b)
    batch.close()
    for p in plans:
        p.close()


@pytest.mark.parametrize("own_dy", [False, True])
def test_list_for_the_tiled_kernel_filled_to_its_capacity(own_dy):
    # 1.5 million windows a period at T0 step 1 (16 items a tile), every period
    # of every wave left to the tiled kernel
    n, kw = 70001, dict(periods_days=np.geomspace(1.0, 9.0, 8), refine_periods=8)
    c = _curve(n, "flat", own_dy, 5)
    got = []
    for flags, chunk in ((0, 4), (2, 0)):
        p = _plan(n, flags, periods_per_chunk=chunk, **kw)
        got.append(gh.gpu_search(p, *c)[1])
        p.close()
    _equal(*got)


def test_chunk_scratch_holds_its_lists():
    # sizes whose folded arrays alone fill 8 GiB but for a few MB
    for n in (52702, 55691, 60409):
        p = _plan(n, 0, periods_days=np.geomspace(1.0, 730.0, 4200))
        before = p.device_bytes()
        p.reserve()
        assert p.device_bytes() - before <= 8 << 30, (n, p.info.periods_per_chunk)
        assert p.info.periods_per_chunk % 152 == 0
        p.close()


def test_tiles_shared_by_unequal_numbers_of_ctas():
    # a wave of periods left to the tiled kernel whose tiles one, two and
    # sixteen CTAs may share
    import torch
    dev = torch.device("cuda:0")
    sizes = (400, 9001, 70001)
    curves = [_curve(n, "flat", False, n) for n in sizes]
    kw = dict(periods_days=np.geomspace(1.0, 9.0, 5), refine_periods=5)
    plans = [_plan(n, 0, **kw) for n in sizes]
    batch = pkg.Batch(plans)
    batch.search(*(torch.as_tensor(np.concatenate([c[k] for c in curves]), device=dev) for k in range(3)),
                 np.cumsum((0,) + sizes).astype(np.int64))
    for i, (n, c) in enumerate(zip(sizes, curves)):
        every = _plan(n, 2, **kw)
        _equal(gh.batch_outputs(batch, i, 5), gh.gpu_search(every, *c)[1])
        every.close()
    batch.close()
    for p in plans:
        p.close()
