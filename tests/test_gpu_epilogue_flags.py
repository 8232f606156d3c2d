"""The flags that place the final epilogue act without FTSP2_PAIR_TILES too: a call
that runs on pairs then takes 256 x 256 tiles, the only ones with a choice."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ft():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2605_08523_gb300 as ft
    return ft


@pytest.mark.parametrize("n,size", [(2200, (256, 256)), (2560, (256, 256)), (300, (128, 64))])
def test_placement_of_the_epilogue(ft, n, size):
    Hd = torch.from_numpy(wl.chain_1d(n, n)).cuda()
    D = {}
    for name, flags in (("default", 0), ("inline", ft.EPI_INLINE), ("deferred", ft.EPI_DEFERRED)):
        s = ft.Solver([n], [0.1], [0.15], ft.ModelSet(), mode="fp16x2", want=3, flags=flags)
        if flags:
            assert s.tile_size() == size, name
        assert s.run(Hd, sync=True) == 0
        D[name] = s.D.clone()
    assert np.isfinite(float(D["default"].sum()))
    assert torch.equal(D["inline"], D["default"]) and torch.equal(D["deferred"], D["default"])


def test_a_recorded_kind_keeps_the_placement(ft):
    ft.ftsp2_autotune_clear()
    n = 2200
    Hd = torch.from_numpy(wl.chain_1d(n, 5)).cuda()
    s = ft.Solver([n], [0.1], [0.15], ft.ModelSet(), mode="fp16x2", want=3, flags=ft.EPI_INLINE)
    choice, single, pair = s.autotune(Hd, reps=1)
    assert s.tile_size() == (256, 256) if choice else s.tile_size()[0] == 128
    ft.ftsp2_autotune_clear()
