"""The inverse transform on its own: a head that runs no band operator, in a plan without an exchange, passes its V coefficients
through, so the output is the inverse of the coefficients the plan holds.  Every form of the last inverse launch, and the three
passes w, h, t on the same grids, against fp64, element by element, and many times over: all buffers that its warps hand to one
another start from other contents each time."""
import numpy as np
import pytest

from oracle import freqformer_oracle as O
from paper_2604_22808_b200 import configs as C

import harness as Hn

pytestmark = pytest.mark.gpu

T_IN_REGISTERS = [(16, 32, 16), (16, 64, 32), (16, 32, 64), (16, 32, 128)]       # every W: 8, 4, 2, 1 lines of w a tile
TWO_AXES = [(16, 16, 16), (32, 32, 16), (32, 32, 32), (64, 16, 64),              # 2, 4, 8, 8 groups of 32 channels an item
            (16, 16, 128), (32, 64, 64)]                                         # 16 channels an item


def _config(grid, heads, d, **more):
    low, mid = tuple(n // 8 for n in grid), tuple(n // 8 + n // 2 for n in grid)
    return C.FFConfig(name="inverse", batch=1, T=grid[0], H=grid[1], W=grid[2], heads=heads, head_dim=d, dtype="bf16", low_cut=low,
                      mid_cut=mid, r=8, b=64, s=8, R=64, m=0, seed=91, timesteps=(500.0,), **more)


@pytest.mark.parametrize("grid", T_IN_REGISTERS + TWO_AXES, ids=lambda g: "x".join(map(str, g)))
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("impl", [0, 4], ids=["default", "three_passes"])
def test_last_launch_of_the_inverse(grid, d, impl):
    import torch
    from paper_2604_22808_b200 import binding as B
    cfg = _config(grid, 3, d)
    plan = B.Plan(cfg)
    plan.set_attention_impl(impl)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    shape = (1, 3) + grid + (d,)
    q, v, other = (torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16) for _ in range(3))
    alloc = torch.zeros(3, dtype=torch.uint8, device="cuda")
    out, want = torch.empty_like(q), None
    for _ in range(40):
        plan.forward(q, q, other, out, alloc=alloc)            # (shared memory and scratch hold another input's values)
        out.fill_(float("nan"))
        plan.forward(q, q, v, out, alloc=alloc)
        want = out.clone() if want is None else want
        assert torch.equal(out, want)
    assert plan.device_status() == 0
    members = O.band_members(cfg.grid, cfg.low_cut, cfg.mid_cut)
    bands = [plan.tap(w).double().cpu().numpy() for w in (B.TAP_SPEC_LOW, B.TAP_SPEC_MID, B.TAP_SPEC_HIGH)]
    for h in range(3):
        spec = np.zeros((cfg.N, d))
        for rows, band in zip(members, bands):
            spec[rows] = band[2, h]
        Hn.assert_close(out[0, h].float().cpu().numpy(), O.inverse_transform(spec.reshape(grid + (d,))), "bf16", f"out head {h}")
    plan.destroy()


@pytest.mark.parametrize("grid,more,two_axes,in_registers", [
    *[(g, {}, True, True) for g in T_IN_REGISTERS], *[(g, {}, True, False) for g in TWO_AXES],
    ((16, 32, 32), {"transform": "haar"}, True, False),        # (its matrix does not fold)
    ((64, 64, 64), {}, False, False), ((16, 32, 48), {}, False, False)], ids=str)
def test_which_launches_a_plan_runs(grid, more, two_axes, in_registers):
    from paper_2604_22808_b200 import binding as B
    plan = B.Plan(_config(grid, 1, 128, **more))
    info = plan.kernel_info()
    assert (info["transform_fused"], info["inverse_t_in_registers"]) == (two_axes, in_registers)
    for impl in (2, 4):                                        # generic transform; three passes
        plan.set_attention_impl(impl)
        info = plan.kernel_info()
        assert (info["transform_fused"], info["inverse_t_in_registers"]) == (False, False)
    plan.destroy()
