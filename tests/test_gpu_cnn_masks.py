"""Loss masks of any value: the mask is counted in integers where it is one and
summed in FP64 elsewhere.  Loss and gradient against the FP64 reference with
the kernels' BF16 parameters and activations, with the bounds that
test_gpu_cnn.py states for masks of zeros and ones (they are relative, and the
mask is a factor of every logit gradient)."""

import numpy as np
import pytest

import paper_2607_00348_gb300 as pkg
from oracle import cnn

from .test_gpu_cnn import _dev, _setup, bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["fractions", "mixed", "small sum", "none"])
def test_gradient_with_any_mask(kind):
    batch = 6
    flat, x, tgt, ones, p_ref = _setup(5, batch)
    rng = np.random.default_rng(6)
    part = np.round(rng.uniform(0.0, 2.0, ones.shape), 3)
    mask = {"fractions": part, "mixed": np.where(rng.random(ones.shape) < 0.5, ones, part),
            "small sum": part * 1e-4, "none": 0.0 * part}[kind].astype(np.float32).astype(float)
    net = pkg.Cnn(8, flat)
    g, loss = net.gradient(_dev(x), _dev(tgt), _dev(mask), batch)
    net.close()
    z_ref, cache = cnn.forward(p_ref, bf16(x), store=bf16)
    loss_ref, dz = cnn.loss_and_dz(z_ref, tgt, mask)
    g_ref = cnn.backward(p_ref, cache, dz)
    assert loss == pytest.approx(loss_ref, rel=1e-3)
    got = cnn.unflatten(g.astype(np.float64))
    for name, _ in cnn.param_shapes():
        ref = g_ref[name]
        np.testing.assert_allclose(got[name], ref, rtol=5e-2, atol=2.5e-2 * np.abs(ref).max(), err_msg=name)
