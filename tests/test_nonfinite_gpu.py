"""A NaN or an infinity in one head reaches the whole of that head's output, as in the definition (the transform spreads
it over a channel's coefficients, the scores over every channel), and no other head's."""
import pytest

from paper_2604_22808_b200 import configs as C
from paper_2604_22808_b200 import inputs as I

import harness as Hn

pytestmark = pytest.mark.gpu

# grid, head_dim, type, summaries, kernel selection
PATHS = [((16, 32, 32), 128, "bf16", 16, 0),      # two axes in one launch
         ((16, 32, 32), 64, "bf16", 16, 4),       # three passes
         ((64, 64, 32), 128, "bf16", 32, 0),      # ... by the size of the plane; one token tile in the exchange
         ((16, 32, 32), 128, "bf16", 40, 0),      # generic exchange
         ((16, 32, 32), 64, "bf16", 0, 0),        # no exchange
         ((13, 20, 33), 128, "bf16", 16, 0), ((13, 20, 33), 64, "bf16", 0, 0),
         ((13, 20, 33), 128, "bf16", 16, 2), ((6, 8, 10), 64, "fp32", 4, 0)]


@pytest.mark.parametrize("grid,d,dtype,m,impl", PATHS, ids=lambda p: str(p).replace(", ", "x"))
@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
def test_nonfinite_input_reaches_the_output(grid, d, dtype, m, impl, value):
    import torch
    from paper_2604_22808_b200 import binding as B
    low = tuple(max(1, n // 8) for n in grid)
    mid = tuple(a + n // 2 for a, n in zip(low, grid))
    cfg = C.FFConfig(name="nonfinite", batch=1, T=grid[0], H=grid[1], W=grid[2], heads=3, head_dim=d, dtype=dtype, low_cut=low,
                     mid_cut=mid, r=8, b=64, s=8, R=64, m=m, seed=71, timesteps=(500.0,))
    qkv = [Hn.to_device(x, cfg) for x in Hn.host_inputs(cfg)]
    plan = B.Plan(cfg, I.router_weights(cfg))
    plan.set_attention_impl(impl)
    alloc = torch.full((3,), 7, dtype=torch.uint8, device="cuda")
    clean = plan.forward(*qkv, torch.empty_like(qkv[0]), alloc=alloc).clone()
    assert torch.isfinite(clean).all()
    for x in qkv:
        keep = x[0, 1, 3, 4, 5, 6].clone()
        x[0, 1, 3, 4, 5, 6] = value
        out = plan.forward(*qkv, torch.empty_like(x), alloc=alloc)
        x[0, 1, 3, 4, 5, 6] = keep
        touched = out[0, 1] if m > 0 or x is not qkv[2] else out[0, 1, ..., 6]      # (only the exchange mixes V's channels)
        assert not torch.isfinite(touched).any()
        assert torch.equal(out[0, 0], clean[0, 0]) and torch.equal(out[0, 2], clean[0, 2])
    plan.destroy()
