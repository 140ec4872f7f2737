"""The FP32 kernel's scratch: what a call reserves covers what its launch addresses,
and never falls as the points grow, in either tile shape.  A captured graph keeps
the buffer's address; a smaller call that needed a larger buffer would free it."""

import ctypes

import pytest


@pytest.mark.parametrize("ff", [0, 1])
@pytest.mark.parametrize("width", [32, 64, 128, 256, 512])
def test_reserved_bytes_cover_the_launch_and_never_fall(nsdf_lib, width, ff):
    import paper_2110_01614_gb300 as nsdf
    arch = nsdf.make_arch(width, 8, activation="relu" if ff else "softplus",
                          ff_freqs=width // 2 if ff else 0)
    plan = (ctypes.c_int64 * 4)()

    def launch(sms, n, nets=0, pt=8, cps=0):
        assert nsdf_lib.nsdf_debug_fp32_plan(ctypes.byref(arch), sms, n, nets, pt, cps, plan) == 0
        assert plan[0] in (4, 8) and plan[1] >= 1 and 0 < plan[2] <= plan[3], (sms, n, nets, pt, cps)
        return plan[0], plan[3]

    # (more SMs stand for more CTAs per SM, which only a GPU can tell)
    for sms in (1, 7, 152, 456):
        sizes = sorted({s + d for s in [16 << k for k in range(15)] + [31 * sms, 32 * sms, 64 * sms,
                                                                       128 * sms, 4800, 8000, 9798]
                        for d in (-1, 0, 1)})
        before, shapes = 0, set()
        for n in sizes:
            shape, single = launch(sms, n)
            shapes.add(shape)
            assert single >= before, (sms, n)
            before = single
        assert shapes == {4, 8}
        for nets in (1, 3, 1000):
            before = 0
            for n in sizes:
                own = [launch(sms, n, nets, pt, cps)[1] for pt in (0, 4, 8) for cps in (0, 1)]
                assert len(set(own)) == 1 and own[0] >= before, (sms, n, nets)
                before = own[0]
                # a single-network call of no more points needs no more
                assert launch(sms, n)[1] <= own[0]


@pytest.mark.parametrize("width,large", [(32, 128), (64, 128), (128, 64), (256, 64), (512, 64)])
def test_grouped_shape_follows_the_bodies(nsdf_lib, width, large):
    """Scenes of bodies that fill few large tiles take the small ones unless told otherwise."""
    import paper_2110_01614_gb300 as nsdf
    arch = nsdf.make_arch(width, 3)
    plan = (ctypes.c_int64 * 4)()

    def shape(total, nets, pt=0):
        assert nsdf_lib.nsdf_debug_fp32_plan(ctypes.byref(arch), 152, total, nets, pt, 0, plan) == 0
        return plan[0]

    assert shape(1000 * 40, 1000) == 4 and shape(1000 * 40, 1000, 8) == 8
    assert shape(1000 * 4 * large, 1000) == 4 and shape(1000 * 4 * large + 1, 1000) == 8
    assert shape(8 * 200000, 8) == 8 and shape(8 * 200000, 8, 4) == 4
    assert shape(2 * 1500, 2) == 4                     # all small tiles fit at once
