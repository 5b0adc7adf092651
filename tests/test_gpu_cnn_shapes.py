"""The proposal network at the edges of its tiles, and time binning of curves
in and out of time order.

Logits and gradients do not depend on what else is in a batch: a curve's
logits are the same bits whatever the batch (its products are added in one
fixed order), and the gradient of a batch is the mean of its curves' gradients
up to the BF16 rounding of the logit gradients, which scale with the batch
(2^-9 relative each: powers of two keep it, so the batches are doubled), and
the FP32 order of the position sums (1e-5).
"""

import numpy as np
import pytest

import paper_2607_00348_gb300 as pkg
from oracle import cnn

pytestmark = pytest.mark.gpu


def _f32(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda:0")


def _forward(net, x):
    import torch
    z = torch.empty((x.shape[0], cnn.N_REG), dtype=torch.float32, device=x.device)
    s = torch.empty_like(z)
    net.forward(x, x.shape[0], logits=z, scores=s)
    return z.cpu().numpy(), s.cpu().numpy()


@pytest.mark.parametrize("batch", [1, 2, 15, 17, 33])
def test_logits_do_not_depend_on_the_batch(batch):
    rng = np.random.default_rng(batch)
    net = pkg.Cnn(40, cnn.flatten(cnn.init_params(3)).astype(np.float32))
    x = _f32(rng.normal(size=(batch, cnn.N_BINS)))
    z, s = _forward(net, x)
    for i in {0, batch // 2, batch - 1}:
        zi, si = _forward(net, x[i:i + 1].contiguous())
        assert np.array_equal(zi[0], z[i]) and np.array_equal(si[0], s[i])
    net.close()


@pytest.mark.parametrize("batch", [1, 8, 32, 64])
def test_gradient_of_a_doubled_batch(batch):
    rng = np.random.default_rng(batch)
    net = pkg.Cnn(2 * batch, cnn.flatten(cnn.init_params(4)).astype(np.float32))
    x = rng.normal(size=(batch, cnn.N_BINS))
    tgt = rng.uniform(size=(batch, cnn.N_REG))
    mask = np.ones((batch, cnn.N_REG))
    g1, l1 = net.gradient(_f32(x), _f32(tgt), _f32(mask), batch)
    twice = lambda a: _f32(np.concatenate([a, a]))  # noqa: E731
    g2, l2 = net.gradient(twice(x), twice(tgt), twice(mask), 2 * batch)
    assert l2 == pytest.approx(l1, rel=1e-12)
    assert np.linalg.norm(g2 - g1) < 1e-5 * np.linalg.norm(g1)
    net.close()


def _times(kind, n, rng):
    t = np.sort(rng.uniform(0.0, 900.0, n))
    if kind == "gaps":
        t[t > 300.0] += 400.0
    if kind == "equal":
        t = np.repeat(t[:max(1, n // 3)], 3)[:n]
        t = np.concatenate([t, np.full(n - t.size, t[-1])])
    if kind == "grid":                                # points on bin edges
        t = np.arange(n) * (900.0 / 4096)
    if kind == "reversed":
        t = t[::-1].copy()
    if kind == "swapped" and n > 2:
        t[n // 2 - 1], t[n // 2] = t[n // 2], t[n // 2 - 1]
    if kind == "late":                                # the last point comes first
        t = np.roll(t, 1)
    return t


@pytest.mark.parametrize("kind", ["sorted", "gaps", "equal", "grid", "reversed", "swapped", "late"])
def test_binning_in_any_order(kind):
    # FP64 sums of at most thousands of points, stored in FP32: 1e-6
    import torch
    rng = np.random.default_rng(7)
    curves = []
    for i, n in enumerate((1, 2, 3, 31, 4097, 9000, 20011)):
        t = _times(kind, n, rng)
        dy = np.full(n, 1e-3) if i % 2 else 1e-3 * rng.uniform(0.5, 1.5, n)
        curves.append((t, 1.0 + rng.normal(0.0, 1e-3, n), dy))
    offs = np.cumsum([0] + [c[0].size for c in curves])
    net = pkg.Cnn(len(curves))
    cat = lambda k: torch.as_tensor(np.concatenate([c[k] for c in curves]), dtype=torch.float64,  # noqa: E731
                                    device="cuda:0")
    for _ in range(2):      # a second call must not see the first one's flags
        x = torch.full((len(curves), cnn.N_BINS), np.nan, dtype=torch.float32, device="cuda:0")
        mean, wsum = torch.empty_like(x), torch.empty_like(x)
        net.bin(cat(0), cat(1), cat(2), offs, x, mean=mean, wsum=wsum)
        for i, (t, y, dy) in enumerate(curves):
            swr, sw = cnn.bin_sums(t, y, dy)
            np.testing.assert_allclose(x[i].cpu().numpy(), cnn.bin_flux(t, y, dy), rtol=1e-6, atol=1e-6)
            np.testing.assert_allclose(wsum[i].cpu().numpy(), sw, rtol=1e-6)
            keep = sw > 0
            np.testing.assert_allclose(mean[i].cpu().numpy()[keep], swr[keep] / sw[keep], rtol=1e-6, atol=1e-9)
    net.close()
