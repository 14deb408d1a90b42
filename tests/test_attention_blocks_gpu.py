"""The fp32 attention at head_dim 64 with few items (less than one an SM) and with several an SM: strided and anchor pattern, fp32 and
bf16 storage, mid items longer than the others."""
import pytest

from paper_2604_22808_b200 import configs as C

from test_parity_gpu import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,heads,dtype,pattern,R", [((5, 14, 17), 2, "fp32", "strided", 40), ((5, 14, 17), 2, "fp32", "anchor", 40),
                                                        ((4, 15, 18), 2, "bf16", "strided", 40), ((4, 28, 45), 14, "fp32", "strided", 200)], ids=str)
def test_blocks_per_sm(grid, heads, dtype, pattern, R):
    low = tuple(max(1, n // 4) for n in grid)
    mid = tuple(min(n, a + n // 2) for n, a in zip(grid, low))
    cfg = C.FFConfig(name="blocks", batch=1, T=grid[0], H=grid[1], W=grid[2], heads=heads, head_dim=64, dtype=dtype, low_cut=low, mid_cut=mid,
                     r=2, b=16, s=3, R=R, m=3, seed=63, mid_pattern=pattern, timesteps=(500.0,))
    _run(cfg, alloc=[7, 6] * (heads // 2), impl=1)
