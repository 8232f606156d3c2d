"""The tile shapes of the tensor-core layers against one another: 128 x 128 tiles
on single CTAs, 256 x 128 ones on pairs, and 256 x 256 ones with either placement
of their epilogue run the same K order per element, so D is the same bit for bit
(the FP64 partial sums are grouped by tile).  Orders at the edges of every tile,
32-column block and K-slice; with one tile per unit the state stays in TMEM
between the layers of a launch, with a launch per layer it does not."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
ORDERS = [1, 31, 32, 33, 64, 65, 127, 129, 191, 257, 300, 385, 513]


@pytest.fixture(scope="module")
def ft():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2605_08523_gb300 as ft
    return ft


def solve(ft, ns, mode, flags, Hd):
    s = ft.Solver(ns, [0.1] * len(ns), [0.15] * len(ns), ft.ModelSet(), mode=mode, want=3, flags=flags)
    s.run(Hd, sync=True)
    return s


@pytest.mark.parametrize("mode", ["fp16x2", "bf16x3", "tf32x3"])
@pytest.mark.parametrize("ns", [ORDERS, [640], [129], [1100, 60]])
def test_shapes_bitwise(ft, mode, ns):
    Hs = [wl.chain_1d(n, 70 + n) if n > 1 else np.array([[0.25]]) for n in ns]
    flat, _ = wl.pack_batch(Hs)
    Hd = torch.from_numpy(flat).cuda()
    # (the flags of a shape also set the accumulation chunks of short batches,
    # the same in all of these)
    base = solve(ft, ns, mode, ft.PAIR_TILES, Hd)
    assert np.isfinite(base.D.cpu().numpy()).all()
    for flags in (ft.PAIR_TILES | ft.LAYER_LAUNCHES, ft.PAIR_TILES | ft.EPI_INLINE, ft.PAIR_TILES | ft.EPI_DEFERRED,
                  ft.SINGLE_TILES, ft.SINGLE_TILES | ft.LAYER_LAUNCHES, ft.SINGLE_TILES | ft.FULL_OPERANDS,
                  ft.PAIR_TILES | ft.FULL_OPERANDS, 0):
        s = solve(ft, ns, mode, flags, Hd)
        assert torch.equal(s.D, base.D), flags
        assert torch.allclose(s.S, base.S, rtol=1e-12, atol=1e-12)
        assert torch.allclose(s.trace, base.trace, rtol=1e-12, atol=1e-12)


@pytest.mark.parametrize("mode", ["fp16x2", "bf16x3", "tf32x3"])
@pytest.mark.parametrize("n", [17, 63, 64, 65, 95, 127, 128, 129, 193, 320, 449, 640])
def test_narrow_tiles_bitwise(ft, mode, n):
    """Single matrices, which run on 128 x 64 tiles by default: the same D, S and trace
    as on pairs, bit for bit, in multi-layer launches (the state in TMEM), with a
    launch per layer, and with the last two layers refined."""
    Hd = torch.from_numpy(wl.chain_1d(n, 90 + n)).cuda()
    for extra in (0, ft.LAYER_LAUNCHES, ft.REFINE2, ft.REFINE2 | ft.REFINE_TC):
        base = solve(ft, [n], mode, ft.PAIR_TILES | extra, Hd)
        s = solve(ft, [n], mode, ft.SINGLE_TILES | extra, Hd)
        assert np.isfinite(base.D.cpu().numpy()).all()
        assert torch.equal(s.D, base.D), extra
        assert torch.equal(s.S, base.S) and torch.equal(s.trace, base.trace), extra
