"""Any grid, many tiles a CTA: every stage, slot and staging area of the passes is used over and over.  Tiles of up to 96 rows and
of more (three and two stages with 128 channels), whole and clipped last tiles.  Coefficients against the generic fp32 kernels,
which are as far from fp64 (a few 2^-24 per axis); a 16-bit coefficient next to the middle of two bf16 numbers may fall to either
side: a bf16 step, 2^-8, of at most 2^-8 of the values.  And the same bits every time, with other values in all buffers between."""
import pytest

from paper_2604_22808_b200 import configs as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,d", [((21, 45, 80), 128), ((9, 100, 66), 128), ((40, 33, 50), 64), ((48, 24, 60), 128)], ids=str)
def test_many_tiles(grid, d):
    _both(grid, d, 4)


# (the middle pass and the band split share their code up to 20 tiles an SM: 6 and 16 of them here, and 25)
@pytest.mark.parametrize("grid,heads", [((5, 33, 20), 8), ((12, 40, 100), 2), ((12, 40, 100), 3)], ids=str)
def test_few_tiles(grid, heads):
    _both(grid, 128, heads)


def _both(grid, d, heads):
    import torch
    from paper_2604_22808_b200 import binding as B
    low, mid = tuple(max(1, n // 8) for n in grid), tuple(n // 8 + n // 2 for n in grid)
    cfg = C.FFConfig(name="tiles", batch=1, T=grid[0], H=grid[1], W=grid[2], heads=heads, head_dim=d, dtype="bf16", low_cut=low, mid_cut=mid,
                     r=8, b=64, s=8, R=64, m=0, seed=93, timesteps=(500.0,))
    plan = B.Plan(cfg)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    q, k, v, other = (torch.randn((1, heads) + grid + (d,), generator=gen, device="cuda").to(torch.bfloat16) for _ in range(4))
    alloc, out = torch.zeros(heads, dtype=torch.uint8, device="cuda"), torch.empty_like(q)
    taps, got = (B.TAP_SPEC_LOW, B.TAP_SPEC_MID, B.TAP_SPEC_HIGH), {}
    for impl in (2, 0, 0, 0):
        plan.set_attention_impl(impl)
        plan.forward(other, other, other, out, alloc=alloc)
        out.fill_(float("nan"))
        plan.forward(q, k, v, out, alloc=alloc)
        new = [plan.tap(w).clone() for w in taps] + [out.clone()]
        assert impl not in got or all(torch.equal(a, b) for a, b in zip(new, got[impl]))
        got[impl] = new
    assert plan.device_status() == 0
    apart = [((a.double() - b.double()).norm() / b.double().norm()).item() for a, b in zip(got[0], got[2])]
    assert apart[0] < 8.0 * 2.0 ** -23 and apart[1] < 2.5e-4 and apart[2] < 2.5e-4 and apart[3] < 2.5e-4, apart
    plan.destroy()
