"""Workspace sizes of the factorisation calls, on the host: what one call made serves every smaller order."""
import ctypes

import pytest

import paper_1907_01063_gb300 as gp


def min_size(n, precision):
    b = ctypes.c_size_t()
    assert gp.capi.gpc_workspace_min_size(n, gp.precision_code(precision), ctypes.byref(b)) == gp.GPC_OK
    return b.value


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_sizes_never_fall_with_the_order(precision):
    orders = list(range(0, 800)) + [4096, 16384, 40960]
    for size in (gp.workspace_size, min_size):
        sizes = [size(n, precision) for n in orders]
        assert all(a <= b for a, b in zip(sizes, sizes[1:]))


def test_room_for_slices_begins_at_one_order():
    # one threshold: no order below it has the room, every order from it on has
    room = [n for n in range(0, 800) if gp.workspace_size(n, "fp64") > min_size(n, "fp64")]
    assert room == list(range(room[0], 800)) and 256 < room[0] < 400


def test_the_mixed_depth_knob_leaves_fp64_sizes_alone():
    # an FP64 call has to fit the workspace it was given before the knob was turned
    old = gp.get_tuning(gp.GPC_TUNE_MIXED_DEFER)
    try:
        sizes = []
        for depth in (1, 6, 8):
            gp.set_tuning(gp.GPC_TUNE_MIXED_DEFER, depth)
            sizes.append([gp.workspace_size(n, "fp64") for n in (300, 321, 700, 1500, 2100, 5000)])
        assert sizes[0] == sizes[1] == sizes[2]
    finally:
        gp.set_tuning(gp.GPC_TUNE_MIXED_DEFER, old)
