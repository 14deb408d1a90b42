"""Where the warps of the tensor-core kernels spend their cycles: `python -m paper_2604_22808_b200.clocks WORKLOAD [--heads N]
[--alloc L,M,H]` builds the library with clocks in its kernels, runs one forward of a workload of `configs.py` and prints, per
role, the cycles of one thread: how often, and how many each time.  The clocks slow the kernels down; the shares count."""
from __future__ import annotations

import argparse
import ctypes
import os

_PASS = {0: "operand makers: wait for copies", 1: "operand makers: work", 2: "issuer: wait for input", 3: "issuer: wait for accumulators",
         4: "epilogue: wait for accumulators", 5: "epilogue: whole tile", 6: "copies: wait for a slot", 7: "epilogue: wait for staging",
         8: "epilogue: read accumulators", 10: "epilogue: fence"}
_PLANE = {0: "phase 1 epilogue: wait for accumulators", 1: "phase 1 epilogue: wait for the plane buffer", 2: "phase 1 epilogue: work",
          3: "phase 2 epilogue: wait for accumulators", 4: "phase 2 epilogue: wait for staging", 5: "phase 2 epilogue: work",
          6: "phase 1 epilogue: hand-over", 7: "issuer 1: wait for input", 8: "issuer 1: wait for accumulators",
          9: "issuer 2: wait for rows", 10: "issuer 2: wait for accumulators", 11: "issuer 2: wait for the second half",
          12: "copies: wait for a slot", 15: "whole kernel"}
_T16 = {0: "copies: wait for a slot", 1: "issuer: wait for input", 2: "issuer: wait for accumulators",
        3: "epilogue: wait for accumulators", 4: "epilogue: wait for staging", 6: "epilogue: stage and send an item",
        7: "whole kernel"}
NAMES = {
    "transform_pass": {16 * m + i: f"{mode}, {what}" for m, mode in enumerate(("first pass", "middle pass", "band split", "last pass"))
                       for i, what in _PASS.items()},
    "transform_plane": {16 * s + i: f"{('forward', 'inverse')[s]}, {what}" for s in range(2) for i, what in _PLANE.items()},
    "transform_t16": {16 * f + i: f"{('inverse', 'forward')[f]}, {what}" for f in range(2) for i, what in _T16.items()},
    "exchange": {0: "copies: wait for a slot", 1: "issuer: wait for tokens", 2: "issuer: wait for P", 3: "issuer: wait for the update buffer",
                 4: "issuer: wait for summaries", 6: "softmax: wait for scores", 7: "softmax: work", 9: "store: wait for the update",
                 10: "store: work", 14: "store: look up positions"},
    "attention": {0: "issuer: Q K", 1: "issuer: P V (with the wait for its second half)", 2: "issuer: wait for the first half of P",
                  3: "issuer: wait for the second half of P", 4: "issuer: a key tile of both streams", 8: "softmax: wait for scores",
                  9: "softmax: masks, load, maximum", 10: "softmax: rescale", 11: "softmax: exponentials, sum, P"},
}


def read(library, kernel: str) -> dict:
    """{what: (times, cycles each)} since the last read, which clears."""
    sums = (ctypes.c_ulonglong * 64)()                         # times in the upper 24 bits, cycles below
    if getattr(library, f"ff_clocks_{kernel}")(sums) != 0:
        raise RuntimeError("could not read the clocks")
    return {name: (sums[i] >> 40, (sums[i] & ((1 << 40) - 1)) / (sums[i] >> 40)) for i, name in NAMES[kernel].items() if sums[i]}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("workload")
    ap.add_argument("--heads", type=int)
    ap.add_argument("--alloc", help="heads per band, e.g. 8,8,8, or `all`: every head runs all three; default: the router's")
    args = ap.parse_args()
    os.environ["FF_LIBRARY_VARIANT"] = "clocks"
    from . import build
    build.build(clocks=True)
    import torch
    from . import binding, configs, inputs
    cfg = configs.BY_NAME[args.workload]
    if args.heads:
        cfg = cfg.scaled(cfg.name, heads=args.heads)
    qkv = [inputs.qkv_full_device(cfg, t, torch.device("cuda:0")) for t in range(3)]
    out = torch.empty_like(qkv[0])
    plan = binding.Plan(cfg, inputs.router_weights(cfg))
    alloc = None
    if args.alloc == "all":
        alloc = [7] * cfg.heads
    elif args.alloc:
        alloc = [1 << band for band, n in enumerate(map(int, args.alloc.split(","))) for _ in range(n)]
    if alloc is not None:
        alloc = torch.tensor(alloc * cfg.batch, dtype=torch.uint8, device="cuda")
    for last in (False, False, True):
        plan.forward(*qkv, out, alloc=alloc, timesteps=[cfg.timesteps[0]] * cfg.batch)
        sums = {kernel: read(binding.library(), kernel) for kernel in NAMES}
    for kernel, rows in sums.items():
        for name, (times, cycles) in rows.items():
            print(f"{kernel:16s} {name:62s} {times:9d} x {cycles:9.0f} cycles")


if __name__ == "__main__":
    main()
