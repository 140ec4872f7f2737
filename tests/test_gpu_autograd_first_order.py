"""Point gradients of a loss of f alone through the autograd Function: the saved
grad f gives what nsdf_backward computes, bit for bit, for FP32 contexts, and
contexts of other precisions still go through it."""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nsdf(nsdf_lib):
    import paper_2110_01614_gb300 as m
    return m


@pytest.mark.parametrize("n", [1, 5000])
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_point_gradient_equals_backward(nsdf, prec, n):
    from paper_2110_01614_gb300.autograd import sdf_query
    arch = synth.Arch(3, 64, 3, -1, 100.0)
    blob = torch.from_numpy(synth.geometric_init(arch, 0)).cuda()
    net = nsdf.NeuralSDF(arch, nsdf.NSDF_FP32 if prec == "fp32" else nsdf.NSDF_BF16)
    pts = torch.from_numpy(synth.body_scale_points(n, 3)).cuda().requires_grad_(True)
    f, g = sdf_query(pts, blob, net)
    a = torch.linspace(-1.0, 1.0, n, device="cuda")
    f.backward(a)
    ref = torch.empty_like(pts)
    nsdf.nsdf_backward(net.ctx, pts.detach(), a, None, None, ref)
    torch.cuda.synchronize()
    assert torch.equal(pts.grad, ref)
    # a loss of f and grad f, or one with trainable weights, is not first order
    pts.grad = None
    f, g = sdf_query(pts, blob, net)
    (f.sum() + g.sum()).backward()
    assert torch.isfinite(pts.grad).all() and not torch.equal(pts.grad, ref)
    net.close()
