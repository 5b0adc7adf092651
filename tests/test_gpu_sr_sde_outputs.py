"""gtls_sr_sde_noalloc with outputs that share memory: SR is written first,
then SDE_raw, then SDE, and what a later one overwrites is not read again."""

import numpy as np
import pytest

from paper_2607_00348_gb300.gtls import sr_sde_noalloc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,window", [(300, 0), (5000, 101), (150001, 0), (400000, 7)])
@pytest.mark.parametrize("shared", ["sde", "sde_raw"])
def test_sr_may_share_an_output(n, window, shared):
    import torch
    rng = np.random.default_rng(n)
    chi2 = torch.as_tensor(1e4 * (1.0 + 1e-3 * rng.random(n)), device="cuda:0")
    sr, raw, sde, one, other = (torch.empty(n, dtype=torch.float64, device="cuda:0") for _ in range(5))
    best = sr_sde_noalloc(chi2, sde, sr=sr, sde_raw=raw, median_window=window)
    want = {"sde": sde, "sde_raw": raw}
    outs = {"sde": other, "sde_raw": None}
    outs[shared] = one
    for _ in range(3):
        got = sr_sde_noalloc(chi2, outs["sde"], sr=one, sde_raw=outs["sde_raw"], median_window=window)
        assert got == best
        assert torch.equal(one, want[shared])
        assert torch.equal(outs["sde"], sde)
