"""Generic fp32-arithmetic kernels at the edges of their tiles: the one-launch transform at and just above the largest
grid it takes, axes of one to three output groups, query and key tiles of 64 with remainders, residue classes shorter
than a tile, windows wider than the band, the anchor pattern, more summaries than a key batch."""
import pytest

from paper_2604_22808_b200 import configs as C

from test_parity_gpu import _run

pytestmark = pytest.mark.gpu

CASES = [
    dict(grid=(4, 18, 32), d=32, dtype="fp32", b=16, s=3, R=70, m=3),       # 2304 positions: the largest one-launch grid
    dict(grid=(5, 21, 22), d=64, dtype="fp32", b=8, s=5, R=1, m=9),         # 2310: separate passes
    dict(grid=(9, 30, 17), d=128, dtype="fp32", b=100, s=2, R=64, m=4),
    dict(grid=(1, 2, 128), d=96, dtype="fp32", b=7, s=40, R=1000, m=1),     # more classes than blocks
    dict(grid=(7, 9, 10), d=32, dtype="bf16", b=16, s=4, R=8, m=40),        # bf16 storage, 120 summaries
    dict(grid=(6, 20, 24), d=96, dtype="bf16", b=32, s=2, R=33, m=5),
    dict(grid=(3, 10, 16), d=96, dtype="bf16", b=16, s=3, R=20, m=2),       # small enough for one warp per query row
    dict(grid=(4, 8, 20), d=128, dtype="fp32", b=5, s=2, R=0, m=2),         # ... with a window of one key
    dict(grid=(5, 16, 24), d=128, dtype="fp32", b=10 ** 9, s=1, R=2 ** 31 - 1, m=2),     # one block, a window of everything
    dict(grid=(6, 20, 24), d=64, dtype="fp32", b=24, s=3, R=16, m=6, mid_pattern="anchor"),
]


@pytest.mark.parametrize("c", CASES, ids=lambda c: "x".join(map(str, c["grid"])) + f"_d{c['d']}_{c['dtype']}")
def test_generic_kernels(c):
    grid = c["grid"]
    low = tuple(max(1, n // 4) for n in grid)
    mid = tuple(min(n, a + n // 2) if n > 1 else 1 for a, n in zip(low, grid))
    cfg = C.FFConfig(name="generic", batch=1, T=grid[0], H=grid[1], W=grid[2], heads=3, head_dim=c["d"], dtype=c["dtype"],
                     low_cut=low, mid_cut=mid, r=2, b=c["b"], s=c["s"], R=c["R"], m=c["m"], seed=61, timesteps=(500.0,),
                     mid_pattern=c.get("mid_pattern", "strided"))
    _run(cfg, alloc=[7, 2, 5], identity_U=False, u_scale=0.2)
    _run(cfg, alloc=[1, 4, 6], impl=3)
