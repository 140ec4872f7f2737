"""The softplus and its slope in nsdf_backward carry FP32 rounding for every
sharpness.  With zero hidden weights the last layer's pre-activations are its
biases b, so one point's gradient gives them as they are: dL/dw_out = h(b) and
dL/db = h'(b) (w_out = 1).  beta b is exact here (powers of two), which leaves
exp (2 ulp), log1p (1 ulp), a division and a sum, or exp and the reciprocal of a
sum: within 5 ulp of the FP64 values."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nsdf(nsdf_lib):
    import paper_2110_01614_gb300 as m
    return m


@pytest.mark.parametrize("width,layers", [(64, 2), (64, 3), (32, 2), (32, 3)])
@pytest.mark.parametrize("beta", [1.0, 16.0, 128.0])
def test_activation_at_fp32_rounding(nsdf, width, layers, beta):
    arch = synth.Arch(3, width, layers, -1, beta)
    net = nsdf.NeuralSDF(arch, nsdf.NSDF_FP32)
    total = synth.n_params(arch)
    b = (np.arange(width) * (96 / width) - 64.0 + 0.375) / beta      # beta b in [-64, 32)
    at_wout = total - 1 - width
    at_b = at_wout - width
    blob = np.zeros(total, np.float32)
    blob[at_b:at_wout] = b
    blob[at_wout:at_wout + width] = 1.0
    net.load(blob)
    P = torch.zeros(1, 4, device="cuda")
    gw = torch.empty(total, device="cuda")
    nsdf.nsdf_backward(net.ctx, P, torch.ones(1, device="cuda"), None, gw, None)
    torch.cuda.synchronize()
    net.close()
    got = gw.cpu().numpy().astype(np.float64)
    u = np.exp(-beta * np.abs(b))
    h = np.maximum(b, 0.0) + np.log1p(u) / beta
    s = np.where(b >= 0, 1.0, u) / (1.0 + u)
    np.testing.assert_allclose(got[at_wout:at_wout + width], h, rtol=5 * 2.0 ** -23)
    np.testing.assert_allclose(got[at_b:at_wout], s, rtol=5 * 2.0 ** -23)
