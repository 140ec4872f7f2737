"""The register-blocked width-64 backward at the edges of its 64-point tiles,
with and without a skip connection, against the FP64 oracle (the bound of the
general kernel's test: 2e-4 of the largest component)."""

import numpy as np
import pytest
import torch

import synth
from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nsdf(nsdf_lib):
    import paper_2110_01614_gb300 as m
    return m


@pytest.mark.parametrize("tangent", [True, False])
@pytest.mark.parametrize("layers,skip", [(2, -1), (2, 1), (3, -1), (3, 1), (3, 2)])
@pytest.mark.parametrize("n", [1, 64, 65, 10007])
def test_matches_oracle(nsdf, layers, skip, n, tangent):
    arch = synth.Arch(3, 64, layers, skip, 100.0)
    blob = synth.geometric_init(arch, 1)
    pts = synth.body_scale_points(n, 2)
    s = synth.Stream(5)
    a = s.normal(n)
    v = s.normal(3 * n).reshape(n, 3) if tangent else np.zeros((n, 3))
    net = nsdf.NeuralSDF(arch, nsdf.NSDF_FP32).load(blob)
    V = None
    if tangent:
        V = torch.zeros(n, 4, device="cuda")
        V[:, :3] = torch.from_numpy(v.astype(np.float32))
    gw = torch.full((synth.n_params(arch),), 7.0, device="cuda")
    gp = torch.full((n, 4), 7.0, device="cuda")
    A = torch.from_numpy(a.astype(np.float32)).cuda()
    P = torch.from_numpy(pts).cuda()
    nsdf.nsdf_backward(net.ctx, P, A, V, gw, gp)
    only_w = torch.full_like(gw, 7.0)
    nsdf.nsdf_backward(net.ctx, P, A, V, only_w, None)
    torch.cuda.synchronize()
    net.close()
    rw, rp = mlp.loss_backward(blob, arch, pts, a, v)
    for got, ref in ((gw.cpu().numpy(), rw), (gp.cpu().numpy()[:, :3], rp)):
        assert np.abs(got - ref).max() <= 2e-4 * np.abs(ref).max()
    assert torch.equal(only_w, gw) and float(gp[:, 3].abs().max()) == 0.0
