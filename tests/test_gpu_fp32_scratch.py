"""A captured graph survives later calls of no more points on its context: they
need no larger scratch, so the buffer that the graph addresses stays."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

EPS = 0.002


@pytest.fixture(scope="module")
def nsdf(nsdf_lib):
    import paper_2110_01614_gb300 as m
    return m


def cloud(n, seed=3):
    return torch.from_numpy(synth.body_scale_points(n, seed)).cuda()


def captured(call):
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        call()
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        call()
    return g


def test_grouped_graph_after_a_smaller_query(nsdf):
    arch = synth.Arch(3, 64, 3, -1, 100.0)
    net = nsdf.NeuralSDF(arch, nsdf.NSDF_FP32, n_nets=3)
    for k in range(3):
        net.load(synth.geometric_init(arch, k), net=k)
    counts = np.array([13000, 7000, 20000], np.int64)
    P = cloud(40000)
    O = torch.from_numpy(np.concatenate([[0], np.cumsum(counts)[:-1]])).cuda()
    C = torch.from_numpy(counts).cuda()
    out, ns = torch.empty_like(P), torch.empty_like(P)
    g = captured(lambda: nsdf.nsdf_query_grouped(net.ctx, P, O, C, 40000, EPS, out, ns))
    g.replay()
    torch.cuda.synchronize()
    ref = out.clone(), ns.clone()
    free = torch.cuda.mem_get_info()[0]
    small = torch.empty(28000, 4, device="cuda")
    for n in (28000, 9700, 1):
        nsdf.nsdf_query(net.ctx, P[:n], small[:n])
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free - small.numel() * 4 - (4 << 20)
    out.zero_(), ns.zero_()
    g.replay()
    nsdf.nsdf_sync_status(net.ctx)
    assert torch.equal(out, ref[0]) and torch.equal(ns, ref[1])
    net.close()


@pytest.mark.parametrize("width,warm,n", [(512, 8000, 4800), (256, 8000, 4800), (64, 40000, 28000)])
def test_capture_after_a_larger_call(nsdf, width, warm, n):
    """Nothing is allocated inside the capture."""
    arch = synth.Arch(3, width, 3, -1, 100.0)
    net = nsdf.NeuralSDF(arch, nsdf.NSDF_FP32).load(synth.geometric_init(arch, 0))
    P = cloud(warm)
    ref, got = torch.empty_like(P), torch.zeros_like(P)
    nsdf.nsdf_query(net.ctx, P, ref)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        nsdf.nsdf_query(net.ctx, P[:n], got[:n])
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(got[:n], ref[:n])
    net.close()


def test_16_bit_graph_after_a_first_order_gradient(nsdf):
    """The FP32 kernel of a 16-bit context has a buffer of its own."""
    arch = synth.Arch(3, 512, 8, 4, 100.0)
    net = nsdf.NeuralSDF(arch, nsdf.NSDF_BF16).load(synth.geometric_init(arch, 0))
    P = cloud(12000)
    ns = torch.zeros_like(P)
    g = captured(lambda: nsdf.nsdf_query(net.ctx, P, ns))
    g.replay()
    torch.cuda.synchronize()
    ref = ns.clone()
    nsdf.nsdf_backward(net.ctx, P, torch.ones(12000, device="cuda"), None, None, torch.empty_like(P))
    ns.zero_()
    g.replay()
    nsdf.nsdf_sync_status(net.ctx)
    assert torch.equal(ns, ref)
    net.close()
