"""Time binning at the edges of what its kernels count and compare: curves of
more points than 32 bits hold, and uncertainties of any bit pattern."""

import numpy as np
import pytest

import paper_2607_00348_gb300 as pkg
from oracle import cnn

pytestmark = pytest.mark.gpu


def _bin(net, t, y, dy, offsets):
    import torch
    n_lc = len(offsets) - 1
    x, mean, wsum = (torch.full((n_lc, cnn.N_BINS), 7.0, dtype=torch.float32, device="cuda:0") for _ in range(3))
    net.bin(t, y, dy, np.asarray(offsets, np.int64), x, mean, wsum)
    return x.cpu().numpy(), mean.cpu().numpy(), wsum.cpu().numpy()


def test_curve_of_more_points_than_32_bits_count():
    import torch
    n, rest = (1 << 31) + 5, 1000
    if torch.cuda.mem_get_info()[0] < 8 * (n + rest) + (2 << 30):
        pytest.skip("less than 20 GB free")
    # one array is times, fluxes and uncertainties: r = 1/2 and w = 4 at every
    # point (sums exact in FP64), one time stamp, so one bin; a usual curve follows
    a = torch.full((n + rest,), 0.5, dtype=torch.float64, device="cuda:0")
    a[n:] = torch.linspace(0.25, 0.75, rest, dtype=torch.float64, device="cuda:0")
    net = pkg.Cnn(2)
    x, mean, wsum = _bin(net, a, a, a, [0, n, n + rest])
    assert x[0, 0] == np.float32(np.sqrt(float(n))) and mean[0, 0] == 0.5 and wsum[0, 0] == np.float32(4.0 * n)
    assert not x[0, 1:].any() and not mean[0, 1:].any() and not wsum[0, 1:].any()
    b = a[n:].clone()
    alone = _bin(net, b, b, b, [0, rest])
    for got, want in zip((x, mean, wsum), alone):
        assert np.array_equal(got[1], want[0])
    net.close()


@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("bits", [-1, 0x7ff8000000000000])
def test_uncertainty_that_is_no_number(bits, ordered):
    # sum w is NaN in the point's bin, whose values are then 0, whatever the
    # NaN's bits; the other bins are those of the curve without the point
    import torch
    n, k = 640, 321
    t = np.linspace(0.0, 10.0, n)
    y = 1.0 + np.random.default_rng(1).normal(0.0, 1e-3, n)
    dy = np.full(n, 1e-3)
    dy[k] = np.array([bits], np.int64).view(np.float64)[0]
    keep = np.arange(n) != k
    order = np.arange(n) if ordered else np.roll(np.arange(n), 77)
    dev = [torch.as_tensor(np.concatenate([a[order], a[keep]]), device="cuda:0") for a in (t, y, dy)]
    net = pkg.Cnn(2)
    x, mean, wsum = _bin(net, *dev, [0, n, 2 * n - 1])
    net.close()
    b = int(np.floor(t[k] / 10.0 * cnn.N_BINS))
    assert np.isnan(wsum[0, b]) and x[0, b] == 0.0 and mean[0, b] == 0.0
    others = np.arange(cnn.N_BINS) != b
    for a in (x, mean, wsum):
        np.testing.assert_allclose(a[0, others], a[1, others], rtol=1e-6, atol=0)
