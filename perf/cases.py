"""What a user of this library has it do, as cases that can be timed.

Kinds of work (``case["kind"]``):

* ``search``  one light curve through ``Plan.search`` (device arrays) or
  ``Plan.search_host`` (host arrays), with every per-period output;
* ``batch``   many light curves, one plan each, through ``Batch.search``;
* ``score``   the period-proposal network on light curves: time binning and
  the forward pass;
* ``forward`` the network alone on inputs that are binned already;
* ``train``   loss and gradient of one training batch of the network;
* ``sr_sde``  SR, SDE_raw and SDE of a chi2(P) spectrum that the caller owns.

Light curves are Kepler-like: a regular cadence with quarter gaps and random
dropouts (or none), white noise with 30 % of red noise, sometimes a transit.
Every curve of a case has the number of points and the baseline that the case
names, whatever the seed.
"""

import math

import numpy as np
import torch

import paper_2607_00348_gb300 as gtls
from paper_2607_00348_gb300 import proposal
from paper_2607_00348_gb300.gtls import sr_sde_noalloc

DAY = 86400.0
GM_SUN = 1.3271244e20
R_SUN = 6.957e8
SPECTRA = ("chi2", "dur_idx", "t0_idx", "depth", "t0", "sr", "sde_raw", "sde")
BEST_FLOATS = ("period", "duration_days", "t0", "depth", "sde", "chi2", "chi2_min", "chi2_0", "snr")
BEST_INTS = ("period_idx", "dur_idx", "dur_points", "t0_idx", "uniform_dy", "refined")

SEARCH = dict(kind="search", n=0, days=0.0, pmin=0.5, pmax=0.0, oversampling=3.0, dt0=0.05, k_min=20.05, k_max=620.84,
              q_cap=0.15, refine=0, dy="uniform", gaps=True, host=False, ppm=104.0)
BATCH = dict(SEARCH, kind="batch", count=0, n_max=0)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # a few nights of ground-based photometry, searched from host arrays: the smallest call
        dict(SEARCH, name="search_tiny_host", n=257, days=12.0, pmin=0.9, pmax=5.0, gaps=False, host=True, ppm=1000.0),
        # one month at 30 min (the 1440-point workload of the tests): latency of a small search
        dict(SEARCH, name="search_month", n=1440, days=29.98, pmax=15.0, gaps=False, ppm=1000.0),
        # four years of Kepler long cadence, whole grid: the workload of the benchmark
        dict(SEARCH, name="search_kepler", n=62363, days=1460.0, pmax=730.0),
        # the shortest curve of the uneven batch with a dy of its own for every point, and the default envelope of TLS
        dict(SEARCH, name="search_dy_per_point", n=20011, days=475.0, dy="point", k_min=41.39, k_max=546.94, q_cap=0.112),
        # two-stage T0 search: the 200 best periods again at T0 step 1
        dict(SEARCH, name="search_refined", n=30001, days=710.0, refine=200),
        # a finer T0 step (the sweep of the benchmark) on two quarters
        dict(SEARCH, name="search_fine_t0", n=8191, days=200.0, dt0=0.01),
        # 3000 days at 30 min, long periods only: the longest curve
        dict(SEARCH, name="search_long_periods", n=144000, days=3000.0, pmin=20.0, pmax=1500.0, gaps=False, ppm=200.0),
        # training targets: curves binned to at most 4096 bins, unit weights, coarser grid
        dict(BATCH, name="batch_binned", count=16, n=3900, n_max=4010, days=1460.0, oversampling=1.0, dy="unit"),
        # triage of many curves by the network, from packed light curves on the device
        dict(name="score_curves", kind="score", count=256, n=20000, n_max=72000),
        # one curve through the network: its latency
        dict(name="forward_one", kind="forward", count=1),
        # one training batch of the proposal network
        dict(name="train_batch", kind="train", count=128),
        # the spectrum of a Kepler-like grid from a caller's own chi2(P)
        dict(name="sr_sde_spectrum", kind="sr_sde", n=199577),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "search", "batch", "batch", "score", "forward", "train", "sr_sde"])
    if kind == "search":
        while True:
            n = _log(rng, 150, 144000)
            days = round(n * 29.4 / 1440.0 / 0.86 * rng.uniform(0.7, 1.3), 3)
            c = dict(SEARCH, n=n, days=days, gaps=rng.random() < 0.7, ppm=float(_log(rng, 50, 2000)),
                     oversampling=rng.choice([1.0, 2.0, 3.0, 3.0]), dt0=rng.choice([0.01, 0.05, 0.05, 0.05, 0.1]),
                     dy=rng.choice(["uniform", "uniform", "point"]), host=rng.random() < 0.3,
                     refine=rng.choice([0, 0, 0, 50, 200]))
            if rng.random() < 0.3:
                c.update(k_min=41.39, k_max=546.94, q_cap=0.112)
            c["pmin"] = round(math.exp(rng.uniform(math.log(max(0.5, 4.0 * days / n)), math.log(days / 8.0))), 3)
            c["pmax"] = round(max(2.0 * c["pmin"], 0.5 * days * rng.uniform(0.3, 1.0)), 3)
            if _affordable(c):
                return c
    if kind == "batch":
        while True:
            n = _log(rng, 200, 24000)
            c = dict(BATCH, count=_log(rng, 2, 64), n=n, n_max=n + rng.randrange(0, n // 2 + 1),
                     days=round(n * 29.4 / 1440.0 / 0.86, 3), oversampling=rng.choice([1.0, 3.0]),
                     dy=rng.choice(["uniform", "mixed", "unit"]), ppm=float(_log(rng, 50, 2000)),
                     refine=rng.choice([0, 0, 50]))
            c["pmin"] = round(max(0.5, 6.0 * c["days"] / n), 3)
            if c["days"] > 8.0 * c["pmin"] and _affordable(c):
                return c
    if kind == "score":
        n = _log(rng, 1000, 60000)
        return dict(kind="score", count=_log(rng, 1, 256), n=n, n_max=n + rng.randrange(0, n // 5 + 1))
    if kind == "sr_sde":
        return dict(kind="sr_sde", n=_log(rng, 200, 500000))
    return dict(kind=kind, count=_log(rng, 1, 256 if kind == "forward" else 128))


def _affordable(c):
    """No dearer than the largest listed searches: points to fold and windows to sum."""
    w, cap = _search_work(c), _search_work(next(x for x in listed() if x["name"] == "search_kepler"))
    weight = 2.0 if c["dy"] in ("point", "mixed") else 1.0
    return w["periods"] >= 40 and weight * w["sums"] <= 0.8 * cap["sums"] and w["folded"] <= 0.8 * cap["folded"]


# ---------------------------------------------------------------------------
# light curves
# ---------------------------------------------------------------------------

def _curve_sizes(c):
    """(points, baseline in days) of every curve of a case."""
    if c["kind"] == "search":
        return [(c["n"], c["days"])]
    span = c["n_max"] - c["n"] + 1
    sizes = [c["n"] + i * 7919 % span for i in range(c["count"])]
    if c["kind"] == "batch" and c["dy"] == "unit":
        return [(n, c["days"]) for n in sizes]          # binned: every curve has the same baseline
    return [(n, c.get("days", 0.0) * n / c["n"] if "days" in c else n * 29.4 / 1440.0 / 0.86) for n in sizes]


def _light_curve(rng, n, days, gaps, ppm, dy):
    """t, y, dy (float64 host arrays) of n points from 0 to `days`."""
    if gaps:
        ncad = max(n + 2, int(math.ceil(n / 0.86)))
        cad = np.arange(ncad) * (days / (ncad - 1))
        inner = np.arange(1, ncad - 1)
        open_ = inner[np.fmod(cad[inner], 91.3125) >= min(3.0, 0.01 * days)]
        if open_.size < n - 2:
            open_ = inner
        keep = np.sort(rng.permutation(open_)[:n - 2])
        t = np.concatenate([[0.0], cad[keep], [days]])
    else:
        t = np.arange(n) * (days / (n - 1))
    sigma = ppm * 1e-6
    white = rng.normal(0.0, sigma / 1.044, n)
    innov = rng.normal(0.0, 0.3 * sigma / 1.044 * math.sqrt(1.0 - 0.81), n + 160)
    red = np.convolve(innov, 0.9 ** np.arange(160), mode="valid")[:n]
    y = 1.0 + white + red
    if rng.random() < 0.5:
        period = math.exp(rng.uniform(math.log(1.0), math.log(max(1.5, days / 4.0))))
        t14 = 111.6 * (period * DAY) ** (1.0 / 3.0) / DAY
        x = np.abs(np.mod(t - rng.uniform(0.0, period) + 0.5 * period, period) - 0.5 * period) / (0.5 * t14)
        mu = np.sqrt(np.clip(1.0 - x * x, 0.0, 1.0))
        y -= np.where(x < 1.0, 2.0 * sigma * (1.0 - 0.4 * (1.0 - mu) - 0.25 * (1.0 - mu) ** 2), 0.0)
    if dy == "point":
        e = sigma * (1.0 + 0.3 * rng.uniform(-1.0, 1.0, n))
    else:
        e = np.full(n, 1.0 if dy == "unit" else sigma)
    return t, y, e


def _light_curves(c, seed):
    rng = np.random.default_rng(seed)
    out = []
    for i, (n, days) in enumerate(_curve_sizes(c)):
        dy = ("point" if i % 2 else "uniform") if c["dy"] == "mixed" else c["dy"]
        out.append(_light_curve(rng, n, days, c["gaps"], c["ppm"], dy))
    return out


def _device(a):
    return torch.as_tensor(a, dtype=torch.float64, device="cuda")


def _packed_curves(c, seed):
    """t, y, dy of all curves on the device, and their offsets (made there: many points)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    sizes = _curve_sizes(c)
    offsets = np.cumsum([0] + [n for n, _ in sizes]).astype(np.int64)
    total = int(offsets[-1])
    ends = torch.as_tensor(offsets[1:], device="cuda")
    which = torch.bucketize(torch.arange(total, device="cuda"), ends, right=True)
    start = torch.as_tensor(offsets[:-1], device="cuda")[which]
    t = (torch.arange(total, device="cuda") - start).double() * (29.4 / 1440.0 / 0.86)
    t += torch.rand(total, generator=g, device="cuda", dtype=torch.float64) * 0.01
    sigma = torch.exp(torch.rand(len(sizes), generator=g, device="cuda", dtype=torch.float64) * 3.7 - 9.9)[which]
    y = 1.0 + sigma * torch.randn(total, generator=g, device="cuda", dtype=torch.float64)
    period = 2.0 + 60.0 * torch.rand(len(sizes), generator=g, device="cuda", dtype=torch.float64)[which]
    y -= torch.where(torch.remainder(t, period) < 0.25, 3.0 * sigma, 0.0)
    return t, y, sigma.clone(), offsets


# ---------------------------------------------------------------------------
# what a program keeps, and one pass
# ---------------------------------------------------------------------------

def _plan(c, n, days):
    pmax = c["pmax"] or 0.5 * days
    return gtls.Plan(gtls.PlanConfig(baseline_days=days, n_points=n, period_min_days=c["pmin"], period_max_days=pmax,
                                     oversampling=c["oversampling"], dt0=c["dt0"], k_min=c["k_min"], k_max=c["k_max"],
                                     q_cap=c["q_cap"], refine_periods=c["refine"]))


def _spectra(n_periods):
    out = {k: torch.empty(n_periods, dtype=torch.int32 if k.endswith("_idx") else torch.float64, device="cuda")
           for k in SPECTRA}
    out["refined"] = torch.empty(n_periods, dtype=torch.int32, device="cuda")
    return out


def _net(count, seed, trained):
    params = np.load(proposal.WEIGHTS)["params"] if trained else proposal.init_params(seed)
    return gtls.Cnn(count, params)


def _net_input(c, seed):
    """Binned curves: unit noise with a few transits."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randn((c["count"], proposal.N_BINS), generator=g, device="cuda")
    phase = torch.arange(proposal.N_BINS, device="cuda")[None, :] % torch.randint(20, 900, (c["count"], 1), generator=g,
                                                                             device="cuda")
    return x + torch.where(phase < 2, 4.0, 0.0) * (torch.rand((c["count"], 1), generator=g, device="cuda") < 0.3), g


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "search":
        t, y, e = _light_curves(c, seed)[0]
        plan = _plan(c, c["n"], c["days"])
        plan.reserve()
        if c["host"]:
            return dict(kind=kind, plan=plan, host=(t, y, e))
        return dict(kind=kind, plan=plan, lc=(_device(t), _device(y), _device(e)), out=_spectra(plan.n_periods))
    if kind == "batch":
        curves = _light_curves(c, seed)
        plans = [_plan(c, n, days) for n, days in _curve_sizes(c)]
        outs = _spectra(sum(p.n_periods for p in plans))
        views, at = [], 0
        for p in plans:
            views.append({k: v[at:at + p.n_periods] for k, v in outs.items()})
            at += p.n_periods
        cat = [_device(np.concatenate([lc[k] for lc in curves])) for k in range(3)]
        offsets = np.cumsum([0] + [lc[0].size for lc in curves]).astype(np.int64)
        return dict(kind=kind, batch=gtls.Batch(plans), lc=cat, offsets=offsets, out=outs, views=views)
    if kind == "score":
        t, y, e, offsets = _packed_curves(c, seed)
        f32 = dict(dtype=torch.float32, device="cuda")
        return dict(kind=kind, net=_net(c["count"], seed, True), lc=(t, y, e), offsets=offsets, count=c["count"],
                    x=torch.empty((c["count"], proposal.N_BINS), **f32), logits=torch.empty((c["count"], proposal.N_REG), **f32),
                    scores=torch.empty((c["count"], proposal.N_REG), **f32))
    if kind == "forward":
        x, _ = _net_input(c, seed)
        f32 = dict(dtype=torch.float32, device="cuda")
        return dict(kind=kind, net=_net(c["count"], seed, True), x=x, count=c["count"],
                    logits=torch.empty((c["count"], proposal.N_REG), **f32), scores=torch.empty((c["count"], proposal.N_REG), **f32))
    if kind == "train":
        x, target, mask = _train_batch(c, seed)
        return dict(kind=kind, net=_net(c["count"], seed, False), x=x, target=target, mask=mask, count=c["count"])
    chi2 = _chi2_spectrum(c, seed)
    return dict(kind=kind, chi2=chi2, sr=torch.empty_like(chi2), raw=torch.empty_like(chi2), sde=torch.empty_like(chi2))


def _train_batch(c, seed):
    x, g = _net_input(c, seed)
    target = torch.rand((c["count"], proposal.N_REG), generator=g, device="cuda") ** 3
    mask = (torch.arange(proposal.N_REG, device="cuda")[None, :] < 122).float().expand(c["count"], -1).contiguous()
    return x, target, mask


def _chi2_spectrum(c, seed):
    """chi2(P) of n periods: noise that follows its neighbours, a slow trend and one deep dip."""
    rng = np.random.default_rng(seed)
    n = c["n"]
    noise = np.convolve(rng.gamma(2.0, 3.0, n + 8), np.ones(9) / 9.0, mode="valid")[:n]
    chi2 = 62000.0 - noise - 6.0 * np.linspace(0.0, 1.0, n) ** 2
    at = rng.integers(0, n)
    chi2[max(0, at - 3):at + 4] -= 150.0
    return _device(chi2)


def _best(res):
    """The candidates of one search or a batch, each field an output of its own (they differ in scale)."""
    rows = res if isinstance(res, list) else [res]
    out = {"best_" + f: np.array([getattr(r, f) for r in rows], np.float64) for f in BEST_FLOATS}
    out["best_at"] = np.array([[getattr(r, f) for f in BEST_INTS] for r in rows], np.int64)
    return out


def run(state):
    kind = state["kind"]
    if kind == "search":
        if "host" in state:
            return _best(state["plan"].search_host(*state["host"]))
        res = state["plan"].search(*state["lc"], per_period=state["out"])
        return dict(_best(res), **state["out"])
    if kind == "batch":
        res = state["batch"].search(*state["lc"], state["offsets"])
        for i, v in enumerate(state["views"]):
            state["batch"].period_outputs(i, v)
        return dict(_best(res), **state["out"])
    if kind == "score":
        state["net"].bin(*state["lc"], state["offsets"], state["x"])
        state["net"].forward(state["x"], state["count"], logits=state["logits"], scores=state["scores"])
        return {k: state[k] for k in ("x", "logits", "scores")}
    if kind == "forward":
        state["net"].forward(state["x"], state["count"], logits=state["logits"], scores=state["scores"])
        return {k: state[k] for k in ("logits", "scores")}
    if kind == "train":
        grad, loss = state["net"].gradient(state["x"], state["target"], state["mask"], state["count"])
        return {"grad": grad, "loss": loss}
    at, top = sr_sde_noalloc(state["chi2"], state["sde"], sr=state["sr"], sde_raw=state["raw"])
    return {"sr": state["sr"], "sde_raw": state["raw"], "sde": state["sde"], "best_at": at, "best_sde": top}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _grid(c, n, days):
    """Trial periods (days, ascending), durations (q, D, T0 step) and each period's first and last duration: the Ofir
    grid and the T14/P grid as include/gtls.h states them."""
    a = (2.0 * math.pi) ** (2.0 / 3.0) / math.pi * R_SUN / math.cbrt(GM_SUN) / (days * DAY * c["oversampling"])
    f_min, f_max = 1.0 / ((c["pmax"] or 0.5 * days) * DAY), 1.0 / (c["pmin"] * DAY)
    c0 = math.cbrt(f_min) - a / 3.0
    count = int(math.ceil((math.cbrt(f_max) - math.cbrt(f_min) + a / 3.0) * 3.0 / a))
    f = (a / 3.0 * np.arange(1, count + 1) + c0) ** 3
    f = f[(f >= f_min * (1.0 - 1e-12)) & (f <= f_max * (1.0 + 1e-12))]
    periods = np.sort(1.0 / (f * DAY))
    p23 = (periods * DAY) ** (-2.0 / 3.0)
    lo, hi = c["k_min"] * p23, np.minimum(c["q_cap"], c["k_max"] * p23)
    q = lo[-1] * 1.1 ** np.arange(0, 1 + int(math.log(hi.max() / lo[-1]) / math.log(1.1)) + 1)
    q = q[q <= hi.max()]
    d = np.minimum(n, np.maximum(1, np.floor(q * n + 0.5))).astype(np.int64)
    st = np.maximum(1, np.floor(d * c["dt0"])).astype(np.int64)
    return periods, q, d, st, np.searchsorted(q, lo, side="left"), np.searchsorted(q, hi, side="right") - 1


def _search_work(c):
    """Periods, points to fold, windows and window-point products of all curves of a case."""
    sizes = _curve_sizes(c)
    out = dict(periods=0, folded=0.0, windows=0.0, sums=0.0, points=0)
    for n, days in sizes if len(sizes) < 3 else [sizes[0], sizes[-1]]:
        share = 1.0 if len(sizes) < 3 else len(sizes) / 2.0
        periods, q, d, st, lo, hi = _grid(c, n, days)
        first = np.concatenate([[True], d[1:] != d[:-1]])     # equal D in a period: the first counts
        wins = np.where(first, -(-n // st), 0)
        cw, cs = np.concatenate([[0.0], np.cumsum(wins)]), np.concatenate([[0.0], np.cumsum(wins * d)])
        out["periods"] += int(share * periods.size)
        out["folded"] += share * float(periods.size) * n
        out["windows"] += share * float((cw[hi + 1] - cw[lo]).sum())
        out["sums"] += share * float((cs[hi + 1] - cs[lo]).sum())
        out["points"] += int(share * n)
    return out


def work(case):
    kind = case["kind"]
    if kind in ("search", "batch"):
        w = _search_work(case)
        outs = 0 if case.get("host") else 60 * w["periods"]
        # the phase of every point at every period (multiply, floor, subtract), and of every window its moving average,
        # depth and chi2: the least that a search has to compute, whichever windows it sums point by point
        return {"bytes": 24 * w["points"] + outs, "flops": 3.0 * w["folded"] + 6.0 * w["windows"]}
    if kind == "sr_sde":
        return {"bytes": 32 * case["n"], "flops": 12 * case["n"]}
    mac, cin, length = 0, 1, proposal.N_BINS
    for taps in proposal.TAPS:
        mac += length * 64 * taps * cin
        cin, length = 64, length // 2
    mac += length * 64 * proposal.N_REG
    params = 4 * (64 * 7 + 5 * 64 * 5 * 64 + 6 * 64 + length * 64 * proposal.N_REG + proposal.N_REG)
    io = 4 * case["count"] * (proposal.N_BINS + 2 * proposal.N_REG)
    if kind == "train":
        return {"bytes": io + 2 * params, "flops": 6.0 * mac * case["count"]}
    points = sum(n for n, _ in _curve_sizes(case)) if kind == "score" else 0
    return {"bytes": 24 * points + io + params, "flops": 2.0 * mac * case["count"] + 8.0 * points}


# ---------------------------------------------------------------------------
# the same in 64 bits, by torch and numpy alone
# ---------------------------------------------------------------------------

def exact(case, seed):
    kind = case["kind"]
    if kind in ("search", "batch"):
        if _search_work(case)["sums"] > 7.0e11:
            return None
        curves, sizes = _light_curves(case, seed), _curve_sizes(case)
        found = [_exact_search(case, n, days, lc) for (n, days), lc in zip(sizes, curves)]
        out = {"best_" + f: np.array([x["best"][f] for x in found]) for f in BEST_FLOATS}
        if not case["host"]:
            out.update({k: torch.cat([x[k] for x in found]) for k in SPECTRA if not k.endswith("_idx")})
        return out
    if kind == "sr_sde":
        sr, raw, sde = _exact_sr_sde(_chi2_spectrum(case, seed))
        return {"sr": sr, "sde_raw": raw, "sde": sde, "best_sde": float(sde.max())}
    if kind == "train":
        x, target, mask = (v.double() for v in _train_batch(case, seed))
        flat = torch.as_tensor(proposal.init_params(seed), device="cuda").double().requires_grad_()
        z = torch.cat([_exact_forward(flat, x[i:i + 16]) for i in range(0, x.shape[0], 16)])
        loss = (mask * (torch.nn.functional.softplus(z) - target * z)).sum() / mask.sum().clamp(min=1.0)
        loss.backward()
        return {"grad": flat.grad, "loss": float(loss.detach())}
    flat = torch.as_tensor(np.load(proposal.WEIGHTS)["params"], device="cuda").double()
    out = {}
    if kind == "score":
        x = _exact_bins(case, seed)
        out["x"] = x
    else:
        x = _net_input(case, seed)[0].double()
    with torch.no_grad():
        z = torch.cat([_exact_forward(flat, x[i:i + 16]) for i in range(0, x.shape[0], 16)])
    return dict(out, logits=z, scores=torch.sigmoid(z))


def _exact_bins(case, seed):
    t, y, e, offsets = _packed_curves(case, seed)
    rows = []
    for a, b in zip(offsets[:-1], offsets[1:]):
        tt, w = t[a:b], 1.0 / e[a:b] ** 2
        at = ((tt - tt.min()) / (tt.max() - tt.min()) * proposal.N_BINS).floor().long().clamp(0, proposal.N_BINS - 1)
        sw = torch.bincount(at, weights=w, minlength=proposal.N_BINS)
        swr = torch.bincount(at, weights=w * (1.0 - y[a:b]), minlength=proposal.N_BINS)
        rows.append(torch.where(sw > 0, swr / sw.clamp(min=1e-300).sqrt(), 0.0))
    return torch.stack(rows)


def _exact_forward(flat, x):
    a, at, cin = x[:, :, None], 0, 1
    for taps, dil in zip(proposal.TAPS, proposal.DILATION):
        w = flat[at:at + 64 * taps * cin].view(64, taps, cin)
        bias = flat[at + 64 * taps * cin:at + 64 * taps * cin + 64]
        at += 64 * taps * cin + 64
        pad, length = (taps - 1) // 2 * dil, a.shape[1]
        ap = torch.nn.functional.pad(a, (0, 0, pad, pad))
        cols = torch.cat([ap[:, k * dil:k * dil + length] for k in range(taps)], dim=2)
        pre = (cols @ w.reshape(64, taps * cin).T + bias).relu()
        a, cin = pre.view(pre.shape[0], length // 2, 2, 64).amax(2), 64
    feat = a.reshape(a.shape[0], -1)
    wh = flat[at:at + proposal.N_REG * feat.shape[1]].view(proposal.N_REG, -1)
    return feat @ wh.T + flat[at + wh.numel():at + wh.numel() + proposal.N_REG]


def _exact_sr_sde(chi2):
    n = chi2.numel()
    sr = torch.where(chi2 > 0, chi2.min() / chi2, 1.0)
    std = (sr - sr.mean()).square().mean().sqrt()
    raw = (sr - sr.mean()) / std if float(std) > 1e-12 else torch.zeros_like(sr)
    h = max(3, 2 * (n // 200) + 1) // 2
    med = torch.empty_like(raw)
    for i in range(n) if n <= 2 * h + 1 else [*range(h), *range(n - h, n)]:
        v = raw[max(0, i - h):i + h + 1]
        med[i] = v.kthvalue((v.numel() - 1) // 2 + 1).values
    if n > 2 * h + 1:
        win, step = raw.unfold(0, 2 * h + 1, 1), max(1, 40_000_000 // (2 * h + 1))
        for a in range(0, win.shape[0], step):
            med[h + a:h + a + step][:win[a:a + step].shape[0]] = win[a:a + step].kthvalue(h + 1, dim=1).values
    return sr, raw, raw - med


def _exact_search(c, n, days, lc):
    """TLS of one curve: fold on the 2^-e day lattice, every window's depth and chi2, the minimum of every period."""
    t, y, dy = (_device(v) for v in lc)
    periods, q, d, st, lo, hi = _grid(c, n, days)
    m, ex = math.frexp(float(periods[-1]))
    e = min(40, 63 - max(1, (n - 1).bit_length()) - (ex - 1 if m == 0.5 else ex))
    d_lat = torch.round((t - t.min()) * 2.0 ** e).long()
    p_lat = torch.as_tensor(np.rint(periods * 2.0 ** e).astype(np.int64), device="cuda")
    r, w = 1.0 - y, 1.0 / dy ** 2
    chi2_0, uniform = float((w * r * r).sum()), bool((dy == dy[0]).all())
    kept = np.zeros((periods.size, q.size), bool)
    for j in range(q.size):
        kept[:, j] = (lo <= j) & (j <= hi) & ((lo == j) | (j == 0 or d[j] != d[j - 1]))
    shape = dict(dtype=torch.float64, device="cuda")
    got = {k: torch.empty(periods.size, **shape) for k in ("chi2", "depth", "t0")}
    dur = torch.zeros(periods.size, dtype=torch.int64, device="cuda")

    def search(sel, steps):
        size = max(1, min(2048, int(1e7 / n)))
        for a in range(0, sel.size, size):
            rows = sel[a:a + size]
            rho = torch.remainder(d_lat[None, :], p_lat[torch.as_tensor(rows, device="cuda")][:, None])
            order = torch.sort(rho, dim=1, stable=True).indices
            fold = lambda v: torch.cat([v[order], v[order][:, :int(d.max())]], dim=1)  # noqa: E731
            total = torch.nn.functional.pad(fold(r).cumsum(1), (1, 0))
            wr, ww = fold(w * r), None if uniform else fold(w)
            best = torch.full((rows.size,), math.inf, **shape)
            at_j, at_s = (torch.zeros(rows.size, dtype=torch.int64, device="cuda") for _ in range(2))
            depth = torch.zeros(rows.size, **shape)
            for j in np.flatnonzero(kept[rows].any(0)):
                on = np.flatnonzero(kept[rows, j])
                dj, sj = int(d[j]), int(steps[j])
                x = (np.arange(dj) + 0.5) / dj
                om = 1.0 - np.sqrt(1.0 - (2.0 * x - 1.0) ** 2)
                s = torch.as_tensor(1.0 - 0.4 * om - 0.25 * om ** 2, device="cuda")
                step = max(1, int(2e8 / (dj * -(-n // sj))))
                for b in range(0, on.size, step):
                    i = torch.as_tensor(on[b:b + step], device="cuda")
                    win = lambda v: v[i, :n + dj - 1].unfold(1, dj, sj)  # noqa: E731
                    dep = ((total[i, dj:n + dj:sj] - total[i, :n:sj]) / s.sum()).clamp(min=0.0)
                    c2 = float(w[0]) * (s * s).sum() if uniform else win(ww) @ (s * s)
                    dchi = dep * (dep * c2 - 2.0 * (win(wr) @ s))
                    v, k = dchi.min(1)
                    better = v < best[i]
                    at = i[better]
                    best[at], at_j[at], at_s[at] = v[better], int(j), k[better] * sj
                    depth[at] = dep.gather(1, k[:, None])[better, 0]
            centre = (at_s + torch.as_tensor(d, device="cuda")[at_j] // 2) % n
            rho_c = rho.gather(1, order.gather(1, centre[:, None]))[:, 0]
            idx = torch.as_tensor(rows, device="cuda")
            got["chi2"][idx], got["depth"][idx], dur[idx] = chi2_0 + best, depth, at_j
            got["t0"][idx] = float(t.min()) + rho_c.double() * 2.0 ** -e

    search(np.arange(periods.size), st)
    sr, raw, sde = _exact_sr_sde(got["chi2"])
    if c["refine"]:
        order = np.lexsort((np.arange(periods.size), -sde.cpu().numpy()))
        search(np.sort(order[:c["refine"]]), np.ones_like(st))
        sr, raw, sde = _exact_sr_sde(got["chi2"])
    got.update(sr=sr, sde_raw=raw, sde=sde)
    b = int(sde.argmax())
    got["best"] = dict(period=periods[b], duration_days=q[int(dur[b])] * periods[b], t0=float(got["t0"][b]),
                       depth=float(got["depth"][b]), sde=float(sde[b]), chi2=float(got["chi2"][b]),
                       chi2_min=float(got["chi2"].min()), chi2_0=chi2_0,
                       snr=math.sqrt(max(0.0, chi2_0 - float(got["chi2"][b]))))
    return got
