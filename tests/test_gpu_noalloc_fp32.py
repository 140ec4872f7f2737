"""nsdf_collide_noalloc in FP32 with few and many slabs in its array, in either tile
shape: the bits of nsdf_collide."""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,layers", [(64, 30), (128, 8), (256, 8), (512, 8)])
def test_bits_do_not_depend_on_the_slabs(nsdf_lib, width, layers):
    import paper_2110_01614_gb300 as nsdf
    arch = synth.Arch(3, width, layers, -1, 100.0)
    net = nsdf.NeuralSDF(arch, nsdf.NSDF_FP32).load(synth.geometric_init(arch, 0))
    pts = torch.from_numpy(synth.body_scale_points(5003, 11)).cuda()
    ref, ref_ns, got, got_ns = (torch.empty_like(pts) for _ in range(4))
    small_slab = 4 * (layers - 1) * width * (32 if width >= 128 else 64)
    nsdf.nsdf_collide(net.ctx, pts, 0.002, ref, ref_ns)
    try:
        for limit in (0, small_slab, 5 * small_slab, 2 * 140 * small_slab):
            nsdf.nsdf_debug_noalloc_limit(limit)
            for n in (1, 2300, 5003):
                got.fill_(7.0), got_ns.fill_(7.0)
                nsdf.nsdf_collide_noalloc(net.ctx, pts[:n], 0.002, got[:n], got_ns[:n])
                nsdf.nsdf_sync_status(net.ctx)
                assert torch.equal(got[:n], ref[:n]) and torch.equal(got_ns[:n], ref_ns[:n])
                assert bool((got[n:] == 7.0).all())
        nsdf.nsdf_debug_noalloc_limit(small_slab - 1)
        with pytest.raises(nsdf.NsdfError) as e:
            nsdf.nsdf_collide_noalloc(net.ctx, pts, 0.002, got)
        assert e.value.status == 8
    finally:
        nsdf.nsdf_debug_noalloc_limit(0)
    net.close()
