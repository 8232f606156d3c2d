"""The Gram reduction of the training at the edges of its blocks: columns around
both slice lengths (m = 4 L + 1 up to 129, and above), chunks of none, one and
several samples, ragged last slices.  Integer entries make every product and sum
exact in FP64, so the result is compared for equality."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("L", [1, 15, 32, 33, 64])
@pytest.mark.parametrize("ns", [1, 63, 65, 64 * 16, 64 * 17 + 5])
def test_gram_exact_on_integers(ft, L, ns):
    rng = np.random.default_rng(100 * L + ns)
    M = rng.integers(-9, 10, (4 * L + 1, ns)).astype(np.float64)
    G = ft.ftsp2_train_normal_equations(torch.from_numpy(M).cuda(), L).cpu().numpy()
    assert np.array_equal(G, M @ M.T)
