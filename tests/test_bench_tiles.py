"""The MMA work that the benchmark counts for a solve: the tiles that touch the upper
triangle, of the shape that the solve runs on."""
import pytest


@pytest.mark.parametrize("tile", [(256, 256), (128, 128), (256, 128), (128, 64)])
@pytest.mark.parametrize("n", [1, 64, 100, 256, 257, 500, 1000, 4096])
def test_tiles_on_the_triangle(n, tile):
    import bench
    rows, cols = tile
    # by definition: tile (I, J) is computed when one of its elements has r <= c, r < n, c < n
    tiles = sum(1 for I in range(-(-n // rows)) for J in range(-(-n // cols)) if I * rows <= (J + 1) * cols - 1)
    flops, layers = bench.hw_flops_per_solve(n, tile, 26, 2, "fp16x2", True)
    assert layers == 26
    assert flops == 2.0 * tiles * rows * cols * n * 2 * (24 * 3 + 2 * 6)
