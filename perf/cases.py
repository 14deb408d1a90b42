"""Performance cases of the FreqFormer attention forward: what a user of this package has it do, through the
package's public entry points (Plan.forward, Plan.forward_host, Plan.forward_projected).

Sizes are the five benchmark workloads and the paper-reference workload of `configs.py`, a small replica of the
kind the tests use, and generic grids: videos whose latent grid is not a power of two along any axis, and fp32
grids of odd sizes.  A case is a dict of plain values; `make_config` turns it into the package's FFConfig."""
import math

import torch

from paper_2604_22808_b200 import binding, configs, inputs

# Parameter sets of the band operators (cut-offs as fractions of an axis, compression r, mid block b and stride s,
# window radius R, summary tokens m), as the benchmark workloads fix them, and the tiny fp32 workload's.
FINE = {"low_div": 8, "r": 8, "b": 64, "s": 8, "R": 256, "m": 16}        # 64K, 256K and 128K workloads
COARSE = {"low_div": 16, "r": 16, "b": 128, "s": 16, "R": 512, "m": 32}  # 1M workload
SMALL = {"low_div": 4, "r": 4, "b": 16, "s": 4, "R": 8, "m": 4}          # tiny workload


def _case(name, entry, dtype, batch, grid, heads, d, par, masks="routed", timestep=500.0, weights_seed=0, smooth=0):
    c = {} if name is None else {"name": name}
    c.update(entry=entry, dtype=dtype, batch=batch, T=grid[0], H=grid[1], W=grid[2], heads=heads, head_dim=d,
             masks=masks, timestep=timestep, weights_seed=weights_seed, smooth=smooth)
    c.update(par)
    return c


# The paper's reference parameterisation (low box half of every axis, mid box 0.79 of it, constant mid degree of
# 256 keys): `low_div` 2 with `mid_frac` stands for its cut-offs.
def _paper(grid):
    low = [n // 2 for n in grid]
    mid = [int(0.8 * n) for n in grid]
    n_mid = mid[0] * mid[1] * mid[2] - low[0] * low[1] * low[2]
    return {"low_div": 2, "mid_frac": 0.8, "r": 4, "b": 32, "s": max(1, round(n_mid / 256)), "R": 32, "m": 8}


def listed():
    return [
        # the smallest call there is: the fp32 correctness grid, one layer of a test or an example
        _case("tiny_fp32", "forward", "fp32", 1, (4, 8, 8), 2, 32, SMALL),
        # a short clip, six heads: launches and host work count as much as the kernels
        _case("clip_16k", "forward", "bf16", 1, (16, 32, 32), 6, 128, FINE, timestep=800.0, weights_seed=11),
        # the headline workload: 64K tokens, 24 heads, early denoising step, the router decides
        _case("grid_64k", "forward", "bf16", 1, (16, 64, 64), 24, 128, FINE, timestep=800.0, weights_seed=1),
        # the same grid under the paper's formal definition: every head runs all three band operators
        _case("grid_64k_all_bands", "forward", "bf16", 1, (16, 64, 64), 24, 128, FINE, masks="all", weights_seed=1),
        # two samples side by side (conditional and unconditional), 128K tokens each
        _case("batch2_128k", "forward", "bf16", 2, (32, 64, 64), 24, 128, FINE, timestep=999.0, weights_seed=4),
        # a long clip with strong low-frequency content, late denoising step, trained (not identity) projections
        _case("smooth_256k", "forward", "bf16", 1, (64, 64, 64), 24, 128, FINE, timestep=200.0, weights_seed=2, smooth=8),
        # the longest clip: a million tokens
        _case("grid_1m", "forward", "bf16", 1, (64, 128, 128), 16, 128, COARSE, weights_seed=3),
        # head_dim 64 with the paper's own band parameters
        _case("paper_ref_64k", "forward", "bf16", 1, (16, 64, 64), 16, 64, _paper((16, 64, 64)), weights_seed=5),
        # a whole attention layer: QKV projections, the forward, output projection
        _case("layer_64k", "projected", "bf16", 1, (16, 64, 64), 24, 128, FINE, timestep=800.0, weights_seed=1),
        # latent grid of a widescreen video, no axis a power of two (76K tokens)
        _case("ragged_76k", "forward", "bf16", 1, (21, 45, 80), 16, 128, FINE, timestep=800.0, weights_seed=21),
        # a full-precision check run on an odd grid, all three operators per head
        _case("odd_fp32_11k", "forward", "fp32", 1, (9, 30, 40), 4, 64, dict(SMALL, R=64, b=32), masks="all", weights_seed=22),
        # activations that live in (pinned) host memory, copied in and out by the call
        _case("host_16k", "host", "bf16", 1, (16, 32, 32), 6, 128, FINE, timestep=800.0, weights_seed=11),
    ]


def make_config(case):
    grid = (case["T"], case["H"], case["W"])
    low = tuple(max(1, n // case["low_div"]) for n in grid)
    if "mid_frac" in case:
        mid = tuple(int(case["mid_frac"] * n) for n in grid)
    else:
        mid = tuple(a + n // 2 for a, n in zip(low, grid))
    mid = tuple(min(n, max(a, b)) for a, b, n in zip(low, mid, grid))
    return configs.FFConfig(name="case", batch=case["batch"], T=case["T"], H=case["H"], W=case["W"], heads=case["heads"],
                            head_dim=case["head_dim"], dtype=case["dtype"], low_cut=low, mid_cut=mid, r=case["r"],
                            b=case["b"], s=case["s"], R=case["R"], m=case["m"], seed=case["weights_seed"],
                            timesteps=(case["timestep"],), smooth_cosines=case["smooth"],
                            smooth_amplitude=3.0 if case["smooth"] else 0.0)


def _bands(cfg):
    n_low = math.prod(cfg.low_cut)
    n_box = math.prod(cfg.mid_cut)
    return n_low, n_box - n_low, cfg.N - n_box


def _attention_flops(cfg, band):
    """4 d operations per scored query-key pair of one head."""
    n_low, n_mid, n_high = _bands(cfg)
    if band == 0:
        n_bar = -(-n_low // cfg.r)
        pairs = n_bar * n_bar
    elif band == 1:
        pairs = n_mid * min(n_mid, max(cfg.b, n_mid / cfg.s))
    else:
        pairs = n_high * min(n_high, 2 * cfg.R + 1)
    return 4.0 * cfg.head_dim * pairs


def work(case):
    """Bytes: inputs read once, the output written once.  Operations: four separable transforms per head by a fast
    algorithm (2.5 N log2 N per channel), the band operators (all three, or for a routed call the average of the
    three: the router gives a head to one band), the exchange with 2m summary tokens, the projections."""
    cfg = make_config(case)
    e = 4 if cfg.dtype == "fp32" else 2
    bh = cfg.batch * cfg.heads
    tensor = float(bh * cfg.N * cfg.head_dim)
    att = sum(_attention_flops(cfg, l) for l in range(3)) / (1 if case["masks"] == "all" else 3)
    flops = 4 * 2.5 * tensor * math.log2(max(2, cfg.N)) + bh * att + 4.0 * 2 * cfg.m * tensor
    nbytes = 4 * tensor * e
    if case["entry"] == "projected":
        D = cfg.heads * cfg.head_dim
        nbytes = 2 * tensor * e + 4.0 * D * D * e
        flops += 4 * 2.0 * tensor * D
    return {"bytes": nbytes, "flops": flops}


def _cost(case):
    w = work(case)
    return w["bytes"] / 6.5e12 + w["flops"] / 1.0e15


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw(rng):
    kind = rng.choices(("grid", "ragged", "paper", "fp32", "projected", "host"), weights=(7, 5, 2, 3, 2, 1))[0]
    seed = rng.randrange(1, 1000)
    timestep = float(rng.choice((999, 800, 750, 500, 250, 200, 1)))
    heads = rng.choice((4, 6, 8, 12, 16, 24))
    masks = rng.choice(("routed", "routed", "routed", "all"))
    if kind == "fp32":
        grid = (rng.randint(2, 12), _log_int(rng, 6, 48), _log_int(rng, 8, 64))
        par = dict(SMALL, R=_log_int(rng, 8, 128), b=rng.choice((16, 32)))
        return _case(None, "forward", "fp32", 1, grid, rng.choice((2, 4, 6)), rng.choice((32, 64, 128)), par, masks, timestep, seed)
    par = rng.choice((FINE, FINE, COARSE))
    if kind == "ragged":
        # latent grids as videos have them: few frames, any height and width
        grid = (rng.randint(5, 40), _log_int(rng, 17, 90), _log_int(rng, 24, 128))
        return _case(None, "forward", "bf16", 1, grid, heads, rng.choice((64, 128, 128)), par, masks, timestep, seed)
    grid = (rng.choice((16, 32, 64)), rng.choice((32, 64, 128)), rng.choice((16, 32, 64, 128)))
    if kind == "paper":
        return _case(None, "forward", "bf16", 1, grid, heads, 64, _paper(grid), masks, timestep, seed)
    if kind == "projected":
        return _case(None, "projected", "bf16", 1, grid, heads, 128, par, masks, timestep, seed)
    if kind == "host":
        return _case(None, "host", "bf16", 1, (16, 32, rng.choice((16, 32, 64))), rng.choice((4, 6, 8)), 128, FINE, masks, timestep, seed)
    return _case(None, "forward", "bf16", rng.choice((1, 1, 1, 2)), grid, heads, 128, par, masks, timestep, seed,
                 rng.choice((0, 0, 8)))


def draw(rng):
    """A case of the same ranges, no dearer than the largest listed one (ragged and fp32 grids: at most 4M and
    64K token-heads, several times the listed ones')."""
    most = max(_cost(c) for c in listed())
    while True:
        c = _draw(rng)
        cfg = make_config(c)
        n = cfg.batch * cfg.heads * cfg.N
        power2 = all(x & (x - 1) == 0 for x in cfg.grid)
        limit = 1 << 16 if cfg.dtype == "fp32" else (1 << 24 if power2 else 1 << 22)
        low, mid, high = _bands(cfg)
        if n <= limit and _cost(c) <= most and min(low, mid, high) > 0:
            return c


def _qkv(cfg, gen, dt):
    """Q, K, V as the path meets them: i.i.d. N(0,1) channels, plus for `smooth` workloads a sum of separable
    cosines of low frequency (amplitude 3, signs per head and channel)."""
    shape = (cfg.batch, cfg.heads, cfg.T, cfg.H, cfg.W, cfg.head_dim)
    wave = None
    if cfg.smooth_cosines:
        f = torch.stack([torch.randint(0, c, (cfg.smooth_cosines,), generator=gen, device="cuda") for c in cfg.low_cut])
        axes = [torch.cos(math.pi * (2.0 * torch.arange(n, device="cuda")[:, None] + 1.0) * f[i][None, :] / (2.0 * n))
                for i, n in enumerate(cfg.grid)]
        wave = torch.einsum("tj,hj,wj->thwj", *axes).reshape(cfg.N, -1)
    out = []
    for _ in range(3):
        x = torch.empty(shape, dtype=dt, device="cuda")
        for b in range(cfg.batch):
            for h in range(cfg.heads):
                v = torch.randn(cfg.N, cfg.head_dim, generator=gen, device="cuda")
                if wave is not None:
                    sign = torch.randint(0, 2, (wave.shape[1], cfg.head_dim), generator=gen, device="cuda").float() * 2 - 1
                    v += cfg.smooth_amplitude * (wave @ sign)
                x[b, h].copy_(v.view(cfg.T, cfg.H, cfg.W, cfg.head_dim))
        out.append(x)
    return out


def prepare(case, seed):
    cfg = make_config(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    dt = torch.float32 if cfg.dtype == "fp32" else torch.bfloat16
    # the router is the model's: its weights belong to the case, the activations to the seed.  Strong low-frequency
    # content comes with summary projections of trained size (rows of norm 1/256), else they are the identity.
    U = inputs.summary_projection(cfg, identity=False, scale=1.0 / 256) if cfg.smooth_cosines else None
    plan = binding.Plan(cfg, inputs.router_weights(cfg), U, host_staging=case["entry"] != "forward")
    state = {"entry": case["entry"], "plan": plan, "timesteps": [case["timestep"]] * cfg.batch, "alloc": None}
    n_masks = cfg.batch * cfg.heads
    if case["entry"] == "projected":
        D = cfg.heads * cfg.head_dim
        state["X"] = torch.randn(cfg.batch, cfg.N, D, generator=gen, device="cuda").to(dt)
        state["Wqkv"] = (torch.randn(3, D, D, generator=gen, device="cuda") / math.sqrt(D)).to(dt)
        state["Wo"] = (torch.randn(D, D, generator=gen, device="cuda") / math.sqrt(D)).to(dt)
        state["out"] = torch.empty_like(state["X"])
    else:
        qkv = _qkv(cfg, gen, dt)
        if case["entry"] == "host":
            qkv = [x.cpu().pin_memory() for x in qkv]
            state["out"] = torch.empty_like(qkv[0], pin_memory=True)
        else:
            state["out"] = torch.empty_like(qkv[0])
        state["Q"], state["K"], state["V"] = qkv
    if case["masks"] == "all":
        all_bands = binding.FF_BAND_LOW | binding.FF_BAND_MID | binding.FF_BAND_HIGH
        state["alloc"] = torch.full((n_masks,), all_bands, dtype=torch.uint8, device="cpu" if case["entry"] == "host" else "cuda")
        if case["entry"] == "host":
            state["alloc"] = state["alloc"].numpy()
        state["timesteps"] = None
    return state


def run(state):
    s, plan = state, state["plan"]
    if s["entry"] == "projected":
        return plan.forward_projected(s["X"], s["Wqkv"], s["Wo"], s["out"], alloc=s["alloc"], timesteps=s["timesteps"])
    if s["entry"] == "host":
        return plan.forward_host(s["Q"], s["K"], s["V"], s["out"], alloc_host=s["alloc"], timesteps=s["timesteps"])
    return plan.forward(s["Q"], s["K"], s["V"], s["out"], alloc=s["alloc"], timesteps=s["timesteps"])


def tolerance(case):
    """bf16 storage rounds band coefficients, operator outputs and the result (2^-9 each); fp32 sums elsewhere."""
    return {"rel": 1e-5, "max": 5e-4} if case["dtype"] == "fp32" else {"rel": 1e-2, "max": 0.1}
