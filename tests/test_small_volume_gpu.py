"""The one-launch transform of grids of up to 256 positions (two outputs a thread) and just above: axes of one, odd, even and 128
positions, more lines than a round takes, fp32 and bf16 storage."""
import pytest

from paper_2604_22808_b200 import configs as C

from test_parity_gpu import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,d,dtype", [((1, 2, 128), 32, "fp32"), ((128, 2, 1), 32, "fp32"), ((3, 5, 7), 64, "fp32"),
                                          ((4, 8, 8), 128, "fp32"), ((2, 3, 43), 96, "fp32"), ((1, 16, 16), 96, "bf16")], ids=str)
def test_small_volume(grid, d, dtype):
    _layer(grid, d, dtype, 2)


# (both sides of the rule: two outputs in several rounds of lines, one block or two an SM and more)
@pytest.mark.parametrize("grid,d,heads", [((3, 9, 9), 64, 2), ((3, 9, 9), 128, 40), ((2, 3, 40), 64, 3), ((4, 8, 8), 96, 24), ((4, 8, 8), 128, 22)], ids=str)
def test_outputs_a_thread(grid, d, heads):
    _layer(grid, d, "fp32", heads)


def _layer(grid, d, dtype, heads):
    low = tuple(max(1, n // 4) for n in grid)
    mid = tuple(min(n, a + n // 2) if n > 1 else 1 for a, n in zip(low, grid))
    cfg = C.FFConfig(name="volume", batch=1, T=grid[0], H=grid[1], W=grid[2], heads=heads, head_dim=d, dtype=dtype, low_cut=low, mid_cut=mid,
                     r=2, b=8, s=3, R=9, m=3, seed=62, timesteps=(500.0,))
    _run(cfg, alloc=[7, 5] * (heads // 2) + [6] * (heads % 2), impl=2)
