"""The forward launch with the second axis in registers (16 or 32 positions along t or h, W <= 64): coefficients of Q, K and V
against fp64, for every number of w lines in a tile (64 / W = 4, 2, 1), either axis, both head_dims; several heads, so that a CTA's
items cross heads and tensors; and many times over, with other values in all buffers in between."""
import numpy as np
import pytest

from oracle import freqformer_oracle as O
from paper_2604_22808_b200 import configs as C

import harness as Hn

pytestmark = pytest.mark.gpu


# (the launch takes 32 positions only where there is work enough for it: more heads)
@pytest.mark.parametrize("grid,heads,d", [((16, 32, 16), 3, 128), ((16, 64, 32), 3, 64), ((16, 32, 64), 3, 128), ((64, 16, 64), 3, 64),
                                          ((32, 64, 64), 3, 128), ((64, 32, 64), 5, 64), ((32, 64, 32), 5, 128), ((32, 64, 16), 10, 128)], ids=str)
def test_forward_fold(grid, heads, d):
    import torch
    from paper_2604_22808_b200 import binding as B
    low, mid = tuple(n // 8 for n in grid), tuple(n // 8 + n // 2 for n in grid)
    cfg = C.FFConfig(name="fold", batch=1, T=grid[0], H=grid[1], W=grid[2], heads=heads, head_dim=d, dtype="bf16", low_cut=low, mid_cut=mid,
                     r=8, b=64, s=8, R=64, m=0, seed=92, timesteps=(500.0,))
    plan = B.Plan(cfg)
    assert plan.kernel_info()["forward_axis_in_registers"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(6)
    q, k, v, other = (torch.randn((1, heads) + grid + (d,), generator=gen, device="cuda").to(torch.bfloat16) for _ in range(4))
    alloc, out = torch.zeros(heads, dtype=torch.uint8, device="cuda"), torch.empty_like(q)
    taps, want = (B.TAP_SPEC_LOW, B.TAP_SPEC_MID, B.TAP_SPEC_HIGH), None
    for _ in range(5):
        plan.forward(other, other, other, out, alloc=alloc)
        plan.forward(q, k, v, out, alloc=alloc)
        got = [plan.tap(w).clone() for w in taps]
        want = got if want is None else want
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert plan.device_status() == 0
    members = O.band_members(cfg.grid, cfg.low_cut, cfg.mid_cut)
    for t, x in enumerate((q, k, v)):
        for h in (0, heads - 1):
            bands = O.split_bands(O.forward_transform(x[0, h].double().cpu().numpy()), members)
            low_got = want[0][t, h].double().cpu().numpy()
            # one intermediate as a bf16 pair and two matrices as pairs (tests/test_precision_gpu.py): below 2^-17 of the norm
            assert np.linalg.norm(low_got - bands[0]) < 2.0 ** -17 * np.linalg.norm(bands[0])
            for got, ref in zip(want[1:], bands[1:]):
                Hn.assert_close(got[t, h].float().cpu().numpy(), ref, "bf16", f"tensor {t} head {h}")
    plan.destroy()


@pytest.mark.parametrize("grid,heads,more,folds", [((16, 32, 16), 1, {}, True), ((32, 64, 32), 3, {}, False), ((32, 64, 32), 4, {}, True),
                                                   ((16, 32, 128), 4, {}, False), ((64, 64, 16), 4, {}, False),
                                                   ((16, 32, 32), 4, {"transform": "haar"}, False), ((16, 32, 48), 4, {}, False)], ids=str)
def test_which_plans_take_it(grid, heads, more, folds):
    from paper_2604_22808_b200 import binding as B
    low, mid = tuple(n // 8 for n in grid), tuple(n // 8 + n // 2 for n in grid)
    plan = B.Plan(C.FFConfig(name="fold", batch=1, T=grid[0], H=grid[1], W=grid[2], heads=heads, head_dim=128, dtype="bf16", low_cut=low,
                             mid_cut=mid, r=8, b=64, s=8, R=64, m=0, seed=92, timesteps=(500.0,), **more))
    assert plan.kernel_info()["forward_axis_in_registers"] == folds
    for impl in (2, 4):                                        # generic transform; three passes
        plan.set_attention_impl(impl)
        assert not plan.kernel_info()["forward_axis_in_registers"]
    plan.destroy()
