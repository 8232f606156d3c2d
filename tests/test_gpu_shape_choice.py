"""The tile shapes taken by default, at sizes where the measured times of the four
shapes lie 4 to 20 % apart (152 SMs).  Each row: order, mode, outputs (1 density,
3 density and entropy), the faster tiles."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MEASURED = [
    (520, "fp16x2", 1, (128, 64)), (520, "tf32x3", 3, (128, 64)), (900, "bf16x3", 3, (128, 64)),
    (1281, "fp16x2", 3, (256, 128)), (1537, "fp16x2", 1, (256, 128)), (2000, "fp16x2", 3, (256, 128)),
    (2000, "tf32x3", 3, (256, 128)), (2200, "fp16x2", 1, (256, 256)), (2200, "tf32x3", 1, (256, 256)),
    (2560, "fp16x2", 1, (256, 256)), (2976, "fp16x2", 1, (128, 128)), (2976, "bf16x3", 1, (128, 128)),
    (3456, "fp16x2", 1, (256, 128)), (3456, "fp16x2", 3, (256, 256)), (3456, "tf32x3", 3, (256, 256)),
    (4100, "fp16x2", 1, (256, 128)), (4400, "fp16x2", 3, (256, 256)), (4400, "bf16x3", 3, (256, 256)),
    (4400, "tf32x3", 3, (256, 256)), (4400, "fp16x2", 1, (256, 128)), (5000, "bf16x3", 1, (256, 256)),
    (5000, "tf32x3", 1, (256, 256)), (8192, "fp16x2", 3, (256, 256))]


@pytest.mark.parametrize("n,mode,want,size", MEASURED)
def test_default_tiles_are_the_faster_ones(n, mode, want, size):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("measured with 152 SMs")
    import paper_2605_08523_gb300 as ft
    from paper_2605_08523_gb300 import _lib
    ft.ftsp2_autotune_clear()
    inst = (_lib.Instance * 1)()
    inst[0].n, inst[0].offset, inst[0].mu, inst[0].kT = n, 0, 0.0, 0.1
    rows, cols = C.c_int(), C.c_int()
    assert ft.lib().ftsp2_tile_size(inst, 1, _lib.MODES[mode], want, 0, C.byref(rows), C.byref(cols)) == 0
    assert (rows.value, cols.value) == size
