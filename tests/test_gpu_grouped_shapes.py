"""FP32 grouped launches of many small bodies and of few: the shape taken by the
bodies' size gives the bits of either shape set by hand."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,nets,size", [(64, 300, 40), (64, 3, 1000), (64, 2, 40000), (32, 200, 130),
                                             (512, 40, 20), (256, 60, 70)])
def test_default_shape_gives_the_same_bits(nsdf_lib, width, nets, size):
    import paper_2110_01614_gb300 as nsdf
    arch = synth.Arch(3, width, 3, -1, 100.0)
    net = nsdf.NeuralSDF(arch, nsdf.NSDF_FP32, n_nets=nets)
    for k in range(nets):
        net.load(synth.geometric_init(arch, k % 5), net=k)
    counts = (size + np.arange(nets) % 7 - 3).astype(np.int64)
    total = int(counts.sum())
    P = torch.from_numpy(synth.body_scale_points(total, 5)).cuda()
    O = torch.from_numpy(np.concatenate([[0], np.cumsum(counts)[:-1]])).cuda()
    C = torch.from_numpy(counts).cuda()

    def run():
        out, ns = torch.full_like(P, 7.0), torch.full_like(P, 7.0)
        nsdf.nsdf_query_grouped(net.ctx, P, O, C, total, 0.002, out, ns)
        nsdf.nsdf_sync_status(net.ctx)
        return out, ns

    ref = run()
    for pt in (4, 8):
        nsdf.nsdf_set_grouped_config(net.ctx, pt, 0)
        got = run()
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    net.close()
