"""The tile sizes that the shape flags force (ftsp2_tile_size): host code, no GPU
needed, since a forced shape is not looked up in the time model."""
import ctypes as C

import pytest


@pytest.fixture(scope="module")
def ft():
    import __graft_entry__ as g
    g.build()
    import paper_2605_08523_gb300 as ft
    return ft


@pytest.mark.parametrize("mode", ["fp16x2", "bf16x3", "tf32x3"])
@pytest.mark.parametrize("ns", [[1], [64], [256], [1501], [8192], [64, 200, 767], [100] * 300])
def test_forced_shapes_whatever_the_size(ft, mode, ns):
    from paper_2605_08523_gb300 import _lib
    inst = (_lib.Instance * len(ns))()
    for i, n in enumerate(ns):
        inst[i].n, inst[i].offset, inst[i].mu, inst[i].kT = n, 0, 0.0, 0.1
    rows, cols = C.c_int(), C.c_int()
    want = {ft.SINGLE_TILES: (128, 128), ft.SINGLE_TILES | ft.HALF_TILES: (128, 64),
            ft.PAIR_TILES: (256, 256), ft.PAIR_TILES | ft.HALF_TILES: (256, 128),
            ft.PAIR_TILES | ft.EPI_INLINE: (256, 256), ft.PAIR_TILES | ft.EPI_DEFERRED: (256, 256)}
    for flags, size in want.items():
        for chains in (1, 2, 3):
            st = ft.lib().ftsp2_tile_size(inst, len(ns), _lib.MODES[mode], chains, flags, C.byref(rows), C.byref(cols))
            assert st == 0 and (rows.value, cols.value) == size, (flags, chains)


def test_tile_size_arguments(ft):
    from paper_2605_08523_gb300 import _lib
    inst = (_lib.Instance * 1)()
    inst[0].n = 64
    rows, cols = C.c_int(7), C.c_int(7)
    call = ft.lib().ftsp2_tile_size
    assert call(inst, 1, _lib.FP32, 3, 0, C.byref(rows), C.byref(cols)) == 0
    assert (rows.value, cols.value) == (0, 0)
    assert call(inst, 0, _lib.FP16X2, 3, ft.PAIR_TILES, C.byref(rows), C.byref(cols)) == _lib.E_ARG
    assert call(inst, 1, _lib.FP16X2, 4, ft.PAIR_TILES, C.byref(rows), C.byref(cols)) == _lib.E_ARG
    assert call(inst, 1, 9, 3, ft.PAIR_TILES, C.byref(rows), C.byref(cols)) == _lib.E_ARG
