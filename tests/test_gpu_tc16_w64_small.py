"""The small-call form of the width-64 tensor-core kernel gives the bits of the
large-call form: small calls (at most a tile per SM) against slices of one large
call, in both precisions, every depth, posed and plain."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nsdf(nsdf_lib):
    import paper_2110_01614_gb300 as m
    return m


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("layers", [2, 3, 5, 7])
def test_small_calls_repeat_the_large_call(nsdf, prec, layers):
    arch = synth.Arch(3, 64, layers, -1, 100.0)
    net = nsdf.NeuralSDF(arch, nsdf.NSDF_BF16 if prec == "bf16" else nsdf.NSDF_FP16)
    net.load(synth.geometric_init(arch, layers))
    T = synth.rigid_transforms(1, seed=3)[0]
    n = 60_001                                          # 469 tiles: the large form
    P = torch.from_numpy(synth.uniform_cube_points(n, 7)).cuda()

    def collide(pts, pose):
        out, ns = torch.empty_like(pts), torch.empty_like(pts)
        hit = torch.empty(pts.shape[0], dtype=torch.uint8, device="cuda")
        net.collide(pts, 0.002, T=pose, out_pts=out, out_n_sdf=ns, out_hit=hit)
        return out, ns, hit

    for pose in (None, T):
        ref = collide(P, pose)
        for m in (1, 127, 128, 129, 4096 + 17, 128 * 100):
            for lo in (0, n - m):
                for a, b in zip(collide(P[lo:lo + m].clone(), pose), ref):
                    assert torch.equal(a, b[lo:lo + m])
    raw = net.query(P, raw_gradient=True)
    assert torch.equal(net.query(P[:500].clone(), raw_gradient=True), raw[:500])
    nsdf.nsdf_sync_status(net.ctx)
    net.close()
