"""What the intermediates of the transform carry, seen in the low band's coefficients, which are kept in fp32: their
error against fp64, relative in the 2-norm, on N(0,1) input."""
import numpy as np
import pytest

from oracle import freqformer_oracle as O
from paper_2604_22808_b200 import configs as C

import harness as Hn

pytestmark = pytest.mark.gpu


def _low_band_error(grid, d, impl=0):
    from paper_2604_22808_b200 import binding as B
    low, mid = tuple(max(1, n // 8) for n in grid), tuple(n // 8 + n // 2 for n in grid)
    cfg = C.FFConfig(name="precision", batch=1, T=grid[0], H=grid[1], W=grid[2], heads=1, head_dim=d, dtype="bf16", low_cut=low,
                     mid_cut=mid, r=8, b=64, s=8, R=64, m=16, seed=81, timesteps=(500.0,))
    qkv = Hn.host_inputs(cfg)
    _, plan = Hn.gpu_forward(cfg, *qkv, None, None, alloc=[7], attention_impl=impl)
    got = plan.tap(B.TAP_SPEC_LOW).double().cpu().numpy()
    plan.destroy()
    members = O.band_members(cfg.grid, cfg.low_cut, cfg.mid_cut)
    want = np.stack([O.split_bands(O.forward_transform(np.asarray(x[0, 0], np.float64)), members)[0] for x in qkv])
    return np.linalg.norm(got[:, 0] - want) / np.linalg.norm(want)


# Two roundings to a bf16 pair, three matrices as pairs and the dropped products of two lo parts in the two passes that
# read pairs: seven errors of up to 2^-18, at most 2^-18 sqrt(7 / 3) = 5.8e-6 if they are uniform and independent (measured
# 5.2e-6 to 6.9e-6).  One byte-form intermediate among them adds an error of up to 2^-17 (measured 8.3e-6 to 1.0e-5).
@pytest.mark.parametrize("grid", [(16, 32, 32), (32, 64, 64), (16, 32, 128), (64, 32, 64)], ids=lambda g: "x".join(map(str, g)))
@pytest.mark.parametrize("d", [64, 128])
def test_pairs_between_the_axes(grid, d):
    assert _low_band_error(grid, d) < 2.0 ** -17


# fp32 grids between the axes, three bf16 parts of matrix and data: as far from fp64 as fp32 arithmetic (which the generic
# kernels do on the same grid: 1.6e-7 to 2.7e-7), a few 2^-24 per axis.
@pytest.mark.parametrize("grid", [(21, 45, 80), (13, 33, 50), (8, 64, 64), (16, 32, 48), (7, 90, 127), (128, 3, 31)],
                         ids=lambda g: "x".join(map(str, g)))
@pytest.mark.parametrize("d", [64, 128])
def test_fp32_between_the_axes_of_any_other_grid(grid, d):
    assert _low_band_error(grid, d) < 4.0 * 2.0 ** -23
    assert _low_band_error(grid, d, impl=2) < 4.0 * 2.0 ** -23


# Planes of 2048 positions go in chunks of 16 channels: every number of coefficients a phase-2 tile can hold (128 / n2 =
# 1, 2, 4, 8); a t axis of 16 has an inverse launch of its own: every W.  Against fp64 and against the separate passes.  The
# latter hand on one byte-form intermediate (2^-16 of the low coefficients' norm); the 16-bit taps differ where a value lies
# that close to the middle of two bf16 numbers, by a bf16 step: share 2^-8 of the values at most, 2^-8 sqrt(2^-8) = 2.5e-4
# of the norm.
@pytest.mark.parametrize("grid", [(128, 128, 16), (64, 64, 32), (32, 64, 64), (16, 32, 128),
                                  (16, 32, 16), (16, 64, 32), (16, 32, 64)], ids=lambda g: "x".join(map(str, g)))
@pytest.mark.parametrize("d", [64, 128])
def test_two_axes_in_one_launch(grid, d):
    import torch
    from paper_2604_22808_b200 import binding as B
    low, mid = tuple(n // 8 for n in grid), tuple(n // 8 + n // 2 for n in grid)
    cfg = C.FFConfig(name="plane", batch=1, T=grid[0], H=grid[1], W=grid[2], heads=1, head_dim=d, dtype="bf16", low_cut=low,
                     mid_cut=mid, r=8, b=64, s=8, R=64, m=16, seed=83, timesteps=(500.0,))
    qkv = Hn.host_inputs(cfg)
    got = []
    for impl in (0, 4):
        out, plan = Hn.gpu_forward(cfg, *qkv, None, None, alloc=[7], attention_impl=impl)
        assert plan.kernel_info()["transform_fused"] == (impl == 0)
        got.append([plan.tap(w).double().clone() for w in (B.TAP_SPEC_LOW, B.TAP_SPEC_MID, B.TAP_SPEC_HIGH)] + [torch.as_tensor(np.asarray(out)).double()])
        plan.destroy()
    apart = [((a - b).norm() / b.norm()).item() for a, b in zip(*got)]
    assert apart[0] < 2.0 ** -16 and apart[1] < 2.5e-4 and apart[2] < 2.5e-4, apart
    assert apart[3] < 2.0 ** -8, apart
    assert _low_band_error(grid, d) < 2.0 ** -17
