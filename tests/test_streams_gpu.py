"""Streams: a forward right behind an event wait reads what the event stands for, whoever waits (the caller, or the
host-buffer call for its own copies), eagerly and in a captured graph."""
import numpy as np
import pytest

from paper_2604_22808_b200 import configs as C
from paper_2604_22808_b200 import inputs as I

import harness as Hn

pytestmark = pytest.mark.gpu

CONFIGS = [C.TINY, C.R64K.scaled("two_axes", heads=3),
           C.R64K.scaled("planes_of_2048", H=16, W=128, low_cut=(2, 2, 16), mid_cut=(10, 10, 80), heads=3),
           C.R64K.scaled("ragged", T=5, H=33, W=20, low_cut=(1, 4, 2), mid_cut=(3, 20, 12), heads=3)]


@pytest.mark.parametrize("cfg", CONFIGS, ids=lambda c: c.name)
@pytest.mark.parametrize("captured", [False, True])
def test_forward_behind_the_callers_event_wait(cfg, captured):
    import torch
    from paper_2604_22808_b200 import binding as B
    plan = B.Plan(cfg, I.router_weights(cfg))
    src = [Hn.to_device(x, cfg) for x in Hn.host_inputs(cfg)]
    alloc = torch.full((cfg.batch * cfg.heads,), 7, dtype=torch.uint8, device="cuda")
    want = plan.forward(*src, torch.empty_like(src[0]), alloc=alloc).clone()
    dst, out = [torch.zeros_like(x) for x in src], torch.zeros_like(src[0])
    slow = torch.zeros(1 << 26, device="cuda")                  # (keeps the side stream busy for a while)
    main, side = torch.cuda.Stream(), torch.cuda.Stream()

    def body():
        """The first forward gives the second one's launch a kernel to follow; the copies come through the side stream."""
        plan.forward(*dst, out, alloc=alloc)
        before, after = torch.cuda.Event(), torch.cuda.Event()
        before.record(main)
        side.wait_event(before)
        with torch.cuda.stream(side):
            for _ in range(4):
                slow.add_(1.0)
            for d, s in zip(dst, src):
                d.copy_(s)
            after.record(side)
        main.wait_event(after)
        plan.forward(*dst, out, alloc=alloc)

    graph = torch.cuda.CUDAGraph()
    if captured:
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=main):
            body()
    for _ in range(5):
        for x in dst + [out]:
            x.zero_()
        torch.cuda.synchronize()
        if captured:
            graph.replay()
        else:
            with torch.cuda.stream(main):
                body()
        torch.cuda.synchronize()
        assert plan.device_status() == 0
        assert torch.equal(out, want)
    del graph
    plan.destroy()


@pytest.mark.parametrize("cfg", CONFIGS[1:], ids=lambda c: c.name)
def test_host_call_equals_the_device_call(cfg):
    """Every group of tensor-heads is transformed after its own copy only: new inputs in every call, into a workspace
    that still holds the last ones."""
    import torch
    from paper_2604_22808_b200 import binding as B
    plan = B.Plan(cfg, I.router_weights(cfg), host_staging=True)
    alloc = torch.full((cfg.batch * cfg.heads,), 7, dtype=torch.uint8)
    src = [Hn.to_device(x, cfg) for x in Hn.host_inputs(cfg)]
    for k in range(4):
        q, kk, v = (src[(i + k) % 3] for i in range(3))
        want = plan.forward(q, kk, v, torch.empty_like(q), alloc=alloc.cuda()).cpu()
        host = [x.cpu().pin_memory() for x in (q, kk, v)]
        out = torch.empty_like(host[0], pin_memory=True)
        for x in src:                                           # (the staged copies of the last call are other tensors)
            plan.forward_host(x.cpu(), x.cpu(), x.cpu(), torch.empty_like(host[0]), alloc_host=alloc.numpy())
        plan.forward_host(*host, out, alloc_host=alloc.numpy())
        assert torch.equal(out, want)
    plan.destroy()


@pytest.mark.parametrize("cfg", CONFIGS[1:], ids=lambda c: c.name)
def test_new_buffers_in_every_call(cfg):
    """The plan's tensor maps are known by their shape: each call puts in its own addresses, in any order, also those of
    other tensors of an earlier call."""
    import torch
    from paper_2604_22808_b200 import binding as B
    plan = B.Plan(cfg, I.router_weights(cfg), host_staging=True)
    alloc = torch.full((cfg.batch * cfg.heads,), 7, dtype=torch.uint8, device="cuda")
    src = [Hn.to_device(x, cfg) for x in Hn.host_inputs(cfg)]
    want = {}
    n = src[0].numel()
    pool = torch.empty(8 * n, dtype=src[0].dtype, device="cuda")
    gen = np.random.default_rng(5)
    for k in range(12):
        slots = gen.permutation(8)[:4]
        order = tuple(gen.integers(0, 3, 3))
        q, kk, v, out = (pool[s * n:(s + 1) * n].view(src[0].shape) for s in slots)
        for dst, i in zip((q, kk, v), order):
            dst.copy_(src[i])
        plan.set_attention_impl(4 if k % 3 == 2 else 0)
        plan.forward(q, kk, v, out, alloc=alloc)
        key = (order, k % 3 == 2)
        if key not in want:
            fresh = B.Plan(cfg, I.router_weights(cfg))
            fresh.set_attention_impl(4 if k % 3 == 2 else 0)
            want[key] = fresh.forward(*(src[i].clone() for i in order), torch.empty_like(src[0]), alloc=alloc).clone()
            fresh.destroy()
        assert torch.equal(out, want[key])
        if k == 6:                                              # (other launch groups, other maps over the same workspace)
            host = [src[i].cpu() for i in order]
            plan.forward_host(*host, torch.empty_like(host[0]), alloc_host=alloc.cpu().numpy())
    plan.destroy()


@pytest.mark.parametrize("batch", [32, 33, 300])
def test_captured_call_keeps_its_timesteps(batch):
    """Up to 32 timesteps travel as arguments of one launch, more in launches of their own; the caller's array may change or
    go once the call has returned."""
    import torch
    from paper_2604_22808_b200 import binding as B
    cfg = C.TINY.scaled("many", batch=batch)
    weights = I.router_weights(cfg)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    q, k, v = (torch.randn((batch, cfg.heads, cfg.T, cfg.H, cfg.W, cfg.head_dim), generator=gen, device="cuda") for _ in range(3))
    ts = np.linspace(0, 999, batch).astype(np.float32)
    plan, one = B.Plan(cfg, weights), B.Plan(C.TINY, weights)
    want = torch.cat([one.forward(*(x[i:i + 1] for x in (q, k, v)), torch.empty_like(q[:1]), timesteps=ts[i:i + 1]) for i in range(batch)])
    out = torch.empty_like(q)
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    gone = ts.copy()
    with torch.cuda.graph(graph, stream=stream):
        plan.forward(q, k, v, out, timesteps=gone)
    gone[:] = -1.0
    for _ in range(2):
        out.zero_()
        plan.tap(B.TAP_PI).zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert (out - want).abs().max() <= 1e-5 * want.abs().max()     # (energies are summed by atomics)
    del graph
    plan.destroy()
    one.destroy()
