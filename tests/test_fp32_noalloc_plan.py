"""The FP32 launch within a fixed amount of scratch: it stays inside, is refused when
not one slab fits, and leaves no SM idle that the smaller tile could use."""

import ctypes

import pytest

MIB = 1 << 20


@pytest.mark.parametrize("width", [32, 64, 128, 256, 512])
@pytest.mark.parametrize("layers", [1, 3, 8, 63])
def test_plan_fits_and_uses_the_sms(nsdf_lib, width, layers):
    import paper_2110_01614_gb300 as nsdf
    arch = nsdf.make_arch(width, layers)
    plan = (ctypes.c_int64 * 3)()

    def launch(n, size, sms=152):
        assert nsdf_lib.nsdf_debug_noalloc_plan(ctypes.byref(arch), sms, n, size, plan) == 0
        return tuple(plan)

    for n in (1, 100, 2300, 5000, 131077):
        for size in (0, 1000, 64 << 10, MIB, 5 * MIB, 32 * MIB):
            for sms in (1, 152):
                shape, grid, used = launch(n, size, sms)
                assert shape in (4, 8) and 0 <= grid <= sms and used <= size
    # with the whole array: every slab of the small tile, or nearly every SM
    shape, grid, used = launch(131077, 32 * MIB)
    small_slab = 4 * max(layers - 1, 1) * width * (32 if width >= 128 else 64)
    assert 8 * grid >= 7 * min(152, 32 * MIB // small_slab)
    assert launch(131077, small_slab) == (4, 1, small_slab)
    assert launch(131077, small_slab - 1)[1] == 0


def test_null_and_bad_arguments(nsdf_lib):
    import paper_2110_01614_gb300 as nsdf
    plan = (ctypes.c_int64 * 3)()
    a = nsdf.make_arch(64, 3)
    assert nsdf_lib.nsdf_debug_noalloc_plan(None, 1, 1, MIB, plan) == 1
    assert nsdf_lib.nsdf_debug_noalloc_plan(ctypes.byref(a), 1, 1, MIB, None) == 1
    assert nsdf_lib.nsdf_debug_noalloc_plan(ctypes.byref(a), 0, 1, MIB, plan) == 1
    assert nsdf_lib.nsdf_debug_noalloc_plan(ctypes.byref(nsdf.make_arch(100, 3)), 1, 1, MIB, plan) == 6
