"""The proposal network at the edges of its tiles.

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

