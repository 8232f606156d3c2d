"""FP32 layers at the edges of their 64 x 64 quadrants, against the oracle's
method-exact density and entropy (the 1e-6 bound of the FP32-class paths): FP32
mode in one ragged call, and as the refinement layers of an FP16X2 solve."""
import numpy as np
import pytest

import workloads as wl
from oracle import pipeline, rescale, tables

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
PRINTED = rescale.Table(tables.PRINTED_B1500, 1500.0, 1.0 / 3.0)
ORDERS = [5, 16, 17, 63, 64, 65, 96, 128, 129, 191, 193, 257]


@pytest.fixture(scope="module")
def ft():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2605_08523_gb300 as ft
    return ft


@pytest.mark.parametrize("mode,flag", [("fp32", ""), ("fp16x2", "REFINE2"), ("tf32x3", "REFINE1")])
def test_quadrant_edges(ft, mode, flag):
    Hs = [wl.chain_1d(n, 40 + n) for n in ORDERS]
    mus = [0.1 if b % 2 else -0.3 for b in range(len(Hs))]
    s = ft.Solver(ORDERS, mus, [0.12] * len(Hs), ft.ModelSet(), mode=mode, want=3,
                  flags=getattr(ft, flag) if flag else 0)
    flat, _ = wl.pack_batch(Hs)
    s.run(torch.from_numpy(flat).cuda(), sync=True)
    for b, (n, H) in enumerate(zip(ORDERS, Hs)):
        ex = pipeline.method_exact(H, mus[b], 0.12, [PRINTED])
        D = s.matrix(b).double().cpu().numpy()
        assert np.array_equal(D, D.T)
        assert np.max(np.abs(D - ex["D"])) < 1e-6, n
        assert abs(float(s.S[b]) - ex["S"]) / n < 1e-6, n
        assert abs(float(s.trace[b, 0]) - np.trace(D)) < 1e-6 * n, n
        assert abs(float(s.trace[b, 1]) - np.sum(D * D)) < 1e-6 * n, n
