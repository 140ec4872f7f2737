"""The output bias's gradient is the plain sum of dL/df: over one tile of the width-64
backward it is a tree of seven sums, so its error stays within 7 half ulps of the sum
of the magnitudes, where one chain would lose every small term (one 1, the others
2^-24)."""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers", [2, 3])
@pytest.mark.parametrize("at", [0, 17, 63])
def test_small_terms_survive(nsdf_lib, layers, at):
    import paper_2110_01614_gb300 as nsdf
    arch = synth.Arch(3, 64, layers, -1, 100.0)
    net = nsdf.NeuralSDF(arch, nsdf.NSDF_FP32).load(synth.geometric_init(arch, 0))
    a = torch.full((64,), 2.0 ** -24)
    a[at] = 1.0
    gw = torch.empty(synth.n_params(arch), device="cuda")
    P = torch.from_numpy(synth.body_scale_points(64, 2)).cuda()
    nsdf.nsdf_backward(net.ctx, P, a.cuda(), None, gw, None)
    torch.cuda.synchronize()
    net.close()
    exact = float(a.double().sum())
    assert abs(float(gw[-1]) - exact) <= 7 * 2.0 ** -24 * exact
