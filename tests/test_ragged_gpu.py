"""Grids with an axis other than 16, 32, 64 and 128, on the tensor-core transform: tiles of fewer than 128 rows, last tiles
that are not full, lines shorter and longer than half a tile, grids smaller than a tile; fp32 between the axes."""
import pytest

from paper_2604_22808_b200 import configs as C

from test_parity_gpu import _run

pytestmark = pytest.mark.gpu

GRIDS = [(3, 5, 7), (9, 33, 17), (1, 12, 128), (7, 127, 6), (21, 20, 24), (16, 32, 48), (2, 65, 66), (128, 3, 31)]


@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "x".join(map(str, g)))
@pytest.mark.parametrize("d", [64, 128])
def test_ragged_grid(grid, d):
    low = tuple(max(1, n // 8) for n in grid)
    mid = tuple(min(n, max(a + n // 2, 1)) for a, n in zip(low, grid))
    cfg = C.FFConfig(name="ragged", batch=1, T=grid[0], H=grid[1], W=grid[2], heads=3, head_dim=d, dtype="bf16",
                     low_cut=low, mid_cut=mid, r=8, b=64, s=8, R=256, m=16, seed=41, timesteps=(500.0,))
    _run(cfg, alloc=[7, 2, 4])
    _run(cfg)


# The exchange writes an fp32 grid there: one and four 16-key chunks (two token tiles), five (tokens read again), more
# summaries than the tensor-core kernel takes, none.
@pytest.mark.parametrize("m", [0, 5, 21, 24, 40])
@pytest.mark.parametrize("d", [64, 128])
def test_ragged_exchange(m, d):
    cfg = C.FFConfig(name="ragged", batch=1, T=6, H=21, W=20, heads=3, head_dim=d, dtype="bf16", low_cut=(2, 4, 5), mid_cut=(4, 13, 14),
                     r=2, b=32, s=3, R=30, m=m, seed=42, timesteps=(500.0,))
    _run(cfg, alloc=[7, 2, 4], identity_U=False, u_scale=0.2)
