"""Kernels that are set up beside the end of their predecessor still see its
writes: chains of calls on one stream, each reading what the one before wrote,
give what the same calls give with a synchronisation between them, directly and
from a captured graph."""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nsdf(nsdf_lib):
    import paper_2110_01614_gb300 as m
    return m


def test_chain_of_steps_and_solves(nsdf):
    nx = 96
    h = 2.0 / (nx - 1)
    arch = synth.Arch(3, 64, 3, -1, 100.0)
    net = nsdf.NeuralSDF(arch, nsdf.NSDF_BF16).load(synth.geometric_init(arch, 0))
    c = torch.linspace(-1.0, 1.0, 32)
    z, y, x = torch.meshgrid(c, c, c, indexing="ij")
    grid = ((x * x + y * y + z * z).sqrt() - 0.55).reshape(-1).contiguous().cuda()
    X0 = torch.from_numpy(synth.cloth_grid(nx, y0=0.5)).cuda()

    def steps(x, prev, count, wait):
        for _ in range(count):
            nsdf.nsdf_cloth_step(x, prev, nx, nx, h, h, 1e4, 9.81, 1e-3)
            wait()
            x, prev = prev, x
            net.collide(x, 0.002, out_pts=x)                      # 72 tiles: the small kernel
            wait()
            nsdf.nsdf_voxel_collide(grid, 32, (-1.0,) * 3, (1.0,) * 3, x, 0.002, x)
            wait()
        return x

    def start():
        prev = X0.clone()
        prev[:, 1] += 2e-3
        return X0.clone(), prev

    ref = steps(*start(), 20, torch.cuda.synchronize).clone()
    assert not torch.equal(ref, X0)
    for _ in range(5):
        assert torch.equal(steps(*start(), 20, lambda: None), ref)
    x, prev = start()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        steps(x, prev, 2, lambda: None)
    for _ in range(10):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(x, ref)
    nsdf.nsdf_sync_status(net.ctx)
    net.close()
