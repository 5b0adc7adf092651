"""SR, SDE_raw, SDE and the argmax on spectra of the library's own, against the
FP64 oracle, at the edges of the reduction's blocks and of the median's.

The sums differ from the oracle's by their order only: about 1e-16 relative,
which the division by the spread of SR (1e-3 or more here) raises to 1e-12;
1e-10 is asserted.  The median is a value of SDE_raw, so SDE follows it.
"""

import numpy as np
import pytest

from oracle import search as osr

pytestmark = pytest.mark.gpu


def _spectrum(kind, n, rng):
    if kind == "smooth":
        return 1000.0 + np.cumsum(rng.normal(0.0, 0.3, n)) - 40.0 * (np.arange(n) == n // 3)
    if kind == "white":
        return 1000.0 + 30.0 * rng.random(n)
    if kind == "levels":                      # many equal values
        return 1000.0 + 5.0 * rng.integers(0, 4, n)
    return np.full(n, 1000.0)                 # flat


@pytest.mark.parametrize("kind", ["smooth", "white", "levels", "flat"])
@pytest.mark.parametrize("n", [1, 2, 31, 1023, 1024, 1025, 4096, 5003, 131071, 200001])
def test_spectrum_matches_the_oracle(kind, n):
    import torch
    from paper_2607_00348_gb300 import gtls as binding
    chi2 = _spectrum(kind, n, np.random.default_rng(n))
    sr, raw, sde = osr.sr_sde(chi2)
    dev = dict(dtype=torch.float64, device="cuda:0")
    out = [torch.full((n,), np.nan, **dev) for _ in range(3)]
    at, top = binding.sr_sde_noalloc(torch.as_tensor(chi2, **dev), out[2], sr=out[0], sde_raw=out[1])
    got = [v.cpu().numpy() for v in out]
    np.testing.assert_allclose(got[0], sr, rtol=1e-14, atol=0)
    np.testing.assert_allclose(got[1], raw, rtol=0, atol=1e-10)
    np.testing.assert_allclose(got[2], sde, rtol=0, atol=1e-10)
    assert top == got[2].max() and at == int(np.argmax(got[2]))


@pytest.mark.parametrize("window", [3, 7, 255, 7999])
def test_other_median_windows(window):
    import torch
    from paper_2607_00348_gb300 import gtls as binding
    n = 20011
    chi2 = _spectrum("smooth", n, np.random.default_rng(window))
    dev = dict(dtype=torch.float64, device="cuda:0")
    sde, raw = torch.empty(n, **dev), torch.empty(n, **dev)
    binding.sr_sde_noalloc(torch.as_tensor(chi2, **dev), sde, sde_raw=raw, median_window=window)
    r = raw.cpu().numpy()
    np.testing.assert_array_equal(sde.cpu().numpy(), r - osr.running_median(r, window))
