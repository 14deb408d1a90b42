"""Summary launch at the edges of its rules: pooled low bands just below and at the length from which the tensor-core
kernel attends them, fewer pooled tokens than segments, segments of one and of several pieces, both storage types."""
import pytest

from paper_2604_22808_b200 import configs as C

from test_parity_gpu import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("low,r,m", [((4, 8, 8), 2, 5), ((4, 8, 8), 3, 1), ((1, 5, 25), 1, 7), ((2, 2, 2), 8, 16), ((1, 3, 43), 1, 32)],
                         ids=["nbar128", "nbar86", "nbar125", "nbar1", "nbar129"])
@pytest.mark.parametrize("d", [64, 128])
def test_low_band_lengths(low, r, m, d):
    cfg = C.FFConfig(name="low", batch=1, T=8, H=16, W=48, heads=3, head_dim=d, dtype="bf16", low_cut=low, mid_cut=(6, 10, 44),
                     r=r, b=32, s=4, R=40, m=m, seed=51, timesteps=(500.0,))
    _run(cfg, alloc=[7, 1, 6], identity_U=False, u_scale=0.2)


@pytest.mark.parametrize("m", [1, 6])
def test_low_band_fp32(m):
    cfg = C.FFConfig(name="low32", batch=2, T=6, H=11, W=23, heads=2, head_dim=96, dtype="fp32", low_cut=(3, 4, 12), mid_cut=(5, 8, 20),
                     r=2, b=16, s=3, R=9, m=m, seed=52, timesteps=(500.0,))
    _run(cfg, alloc=[7, 1, 6, 5], identity_U=False)
