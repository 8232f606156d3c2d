"""Each of the four tile shapes of the tensor-core layers, forced, at the edges of
its tiles, of the 32-column blocks and of the K-slices; the tile tables of large
batches; and the bounded waits of every shape.

A shape changes neither the order of the products of an element nor the blocks that
S and the traces are summed by, so everything is compared bit for bit."""
import time

import numpy as np
import pytest

import workloads as wl
from oracle import pipeline, rescale, tables

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PRINTED = rescale.Table(tables.PRINTED_B1500, 1500.0, 1.0 / 3.0, name="printed")
EDGES = [1, 31, 32, 33, 63, 64, 65, 95, 96, 127, 128, 129, 191, 193, 255, 257, 300, 385, 449, 513]
SIZES = {"single": (128, 128), "single_half": (128, 64), "pair": (256, 256), "pair_half": (256, 128)}


@pytest.fixture(scope="module")
def ft():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2605_08523_gb300 as ft
    return ft


def flag_of(ft, shape):
    f = ft.PAIR_TILES if shape.startswith("pair") else ft.SINGLE_TILES
    return f | (ft.HALF_TILES if shape.endswith("half") else 0)


def matrices(ns, seed):
    return [wl.chain_1d(n, seed + 1000 * i + n) if n > 1 else np.array([[0.25]]) for i, n in enumerate(ns)]


def solve(ft, ns, mode, flags, Hd, want=3):
    s = ft.Solver(ns, [0.1] * len(ns), [0.15] * len(ns), ft.ModelSet(), mode=mode, want=want, flags=flags)
    s.run(Hd, sync=True)
    return s


def same(a, b):
    return torch.equal(a.D, b.D) and torch.equal(a.trace, b.trace) and (a.want == 1 or torch.equal(a.S, b.S))


@pytest.mark.parametrize("mode", ["fp16x2", "bf16x3", "tf32x3"])
@pytest.mark.parametrize("extra", ["", "layers", "full", "refine_fp32", "refine_tc"])
@pytest.mark.parametrize("ns", [EDGES, [65], [129], [640], [1100, 60]], ids=["edges", "65", "129", "640", "1100_60"])
def test_four_shapes_bitwise(ft, mode, extra, ns):
    Hd = torch.from_numpy(wl.pack_batch(matrices(ns, 11))[0]).cuda()
    x = {"": 0, "layers": ft.LAYER_LAUNCHES, "full": ft.FULL_OPERANDS, "refine_fp32": ft.REFINE2,
         "refine_tc": ft.REFINE2 | ft.REFINE_TC}[extra]
    runs = {}
    for shape, size in SIZES.items():
        s = runs[shape] = solve(ft, ns, mode, flag_of(ft, shape) | x, Hd)
        assert s.tile_size() == size
    assert bool(torch.isfinite(runs["pair"].D).all())
    for shape, s in runs.items():
        assert same(s, runs["pair"]), shape


@pytest.mark.parametrize("mode", ["fp16x2", "bf16x3", "tf32x3"])
@pytest.mark.parametrize("ns,want", [([128] * 100, 1), ([96] * 140, 1), ([100] * 60, 3),
                                     ([65 + (37 * i) % 64 for i in range(70)], 3)],
                         ids=["100x128", "140x96", "60x100", "70x65-128"])
def test_one_square_tile_per_cta(ft, mode, ns, want):
    """Batches with one 128 x 128 tile per CTA, which run on those by default in FP16X2
    mode: B read from A's panel, the state in TMEM and the operands staged in the ring."""
    Hs = matrices(ns, 23)
    Hd = torch.from_numpy(wl.pack_batch(Hs)[0]).cuda()
    s = solve(ft, ns, mode, 0 if mode == "fp16x2" else ft.SINGLE_TILES, Hd, want)
    assert s.tile_size() == (128, 128)
    for flags in (ft.PAIR_TILES, 0, ft.SINGLE_TILES | ft.LAYER_LAUNCHES, ft.SINGLE_TILES | ft.HALF_TILES):
        assert same(s, solve(ft, ns, mode, flags, Hd, want)), flags
    for b in (0, len(ns) // 2, len(ns) - 1):
        ex = pipeline.method_exact(Hs[b], 0.1, 0.15, [PRINTED])
        D = s.matrix(b).double().cpu().numpy()
        assert np.max(np.abs(D - ex["D"])) < 1e-6


@pytest.mark.parametrize("mode,flags", [("fp16x2", ""), ("fp16x2", "pair"), ("fp16x2", "single_half"),
                                        ("tf32x3", "pair_half"), ("fp16x2", "refine_fp32"), ("fp32", "")])
@pytest.mark.parametrize("nb", [2049, 3100])
def test_tile_tables_past_the_sorted_batches(ft, mode, flags, nb):
    """More instances than the tile tables sort: the same results as in two batches."""
    r = np.random.default_rng(nb)
    ns = [int(n) for n in r.integers(1, 90, nb)]
    ns[7], ns[nb - 1], ns[nb // 2] = 300, 257, 129
    Hs = matrices(ns, 5)
    x = ft.REFINE2 if flags == "refine_fp32" else flag_of(ft, flags) if flags else 0
    whole = solve(ft, ns, mode, x, torch.from_numpy(wl.pack_batch(Hs)[0]).cuda())
    cut, at = nb // 2 + 1, 0
    for part in (slice(0, cut), slice(cut, nb)):
        p = solve(ft, ns[part], mode, x, torch.from_numpy(wl.pack_batch(Hs[part])[0]).cuda())
        k = p.D.numel()
        assert torch.equal(whole.D[at:at + k], p.D)
        assert torch.equal(whole.S[part], p.S) and torch.equal(whole.trace[part], p.trace)
        at += k
    assert at == whole.D.numel() and all(int(q["status"]) == 0 for q in whole.records())


@pytest.mark.parametrize("mode", ["fp16x2", "tf32x3"])
@pytest.mark.parametrize("dims", [(8, 8, 16), (8, 16, 16)], ids=["1024", "2048"])
@pytest.mark.parametrize("shape", list(SIZES))
def test_stalled_dependency_of_every_shape(ft, mode, dims, shape):
    """n = 1024: one tile per unit where the tiles are smaller than 256 x 256 (the state
    in TMEM); n = 2048: several.  The wait runs out on the device, is reported in every
    record, and the next call is undisturbed."""
    H = wl.lattice_3d(dims, 0)
    n = H.shape[0]
    Hd = torch.from_numpy(H.ravel().copy()).cuda()
    s = ft.Solver([n], [0.0], [0.1], ft.ModelSet(), mode=mode, want=3, flags=flag_of(ft, shape))
    assert s.run(Hd, sync=True) == 0
    D0, S0, T0 = s.D.clone(), s.S.clone(), s.trace.clone()
    default = ft.wait_limit_ns()
    ft.set_wait_limit_ns(2_000_000)
    ft.debug_stall_layer(5)
    try:
        t0 = time.perf_counter()
        st = s.run(Hd, sync=True)
        dt = time.perf_counter() - t0
    finally:
        ft.debug_stall_layer(-1)
        ft.set_wait_limit_ns(default)
    assert st == -6 and np.all(s.records()["status"] == -6)
    assert dt < 5.0, dt
    assert s.run(Hd, sync=True) == 0
    assert torch.equal(s.D, D0) and torch.equal(s.S, S0) and torch.equal(s.trace, T0)
