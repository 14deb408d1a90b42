"""The hand-over of two staging buffers between the warps that fill them and the one that sends them out
(csrc/ff_two_buffers.h): its functions, compiled for the host, in a model that takes every order of the warps.  No store goes
out before all parts of its step are written, no part is written while a store still reads the buffer, nobody waits for good."""
import ctypes
import os
import shutil
import subprocess
from types import SimpleNamespace

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2604_22808_b200", "csrc")
FUNCTIONS = ("buffer", "full", "full_parity", "waits_free", "free_parity")
WARPS, STEPS = 4, 9                     # warp 0 issues; all parities come back after four steps

# One full barrier for both buffers: what the hand-over must not be.
ONE_BARRIER = SimpleNamespace(buffer=lambda n: n & 1, full=lambda n: 0, full_parity=lambda n: n & 1, waits_free=lambda n: n >= 2,
                              free_parity=lambda n: n & 1)


@pytest.fixture(scope="module")
def handover(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    assert cxx, "no C++ compiler"
    folder = tmp_path_factory.mktemp("two_buffers")
    source, lib = str(folder / "shim.cpp"), str(folder / "shim.so")
    with open(source, "w") as f:
        f.write('#include "ff_two_buffers.h"\nextern "C" {\n')
        for name in FUNCTIONS:
            f.write(f"int {name}(unsigned n) {{ return (int)FFTwoBuffers::{name}(n); }}\n")
        f.write("}\n")
    subprocess.run([cxx, "-shared", "-fPIC", "-I", CSRC, "-o", lib, source], check=True)
    return SimpleNamespace(**{name: getattr(ctypes.CDLL(lib), name) for name in FUNCTIONS})


def explore(h):
    """Depth-first through all states; returns what went wrong, or None.  A state: each warp's step and action; arrivals and
    ended phases of the barriers (0, 1: full, 2: free); who wrote which step into which buffer last; the stores (by step) still
    reading; how many have been issued."""
    def passes(bars, b, parity):                     # a parity wait: the phase of that parity has ended
        return bars[b][1] & 1 != parity

    def arrive(bars, b, of):
        n, phase = bars[b][0] + 1, bars[b][1]
        return bars[:b] + ((0, phase + 1) if n == of else (n, phase),) + bars[b + 1:]

    start = (tuple((0, 0) for _ in range(WARPS)), ((0, 0),) * 3, ((None,) * WARPS,) * 2, (), 0)
    seen, todo = {start}, [start]
    while todo:
        pcs, bars, bufs, reading, issued = todo.pop()
        after = []
        if reading:                                  # the oldest store has read its buffer
            after.append((pcs, bars, bufs, reading[1:], issued))
        for w, (n, act) in enumerate(pcs):
            if n == STEPS:
                continue
            nb, nf, nr, ni = bars, bufs, reading, issued
            if act == 0:
                if h.waits_free(n) and w == 0:
                    if any(s <= n - 2 for s in reading):
                        continue
                    nb = arrive(bars, 2, 1)
            elif act == 1:
                if h.waits_free(n) and not passes(bars, 2, h.free_parity(n)):
                    continue
            elif act == 2:
                b = h.buffer(n)
                if any(h.buffer(s) == b for s in reading):
                    return f"warp {w} writes step {n} into a buffer that is being read"
                nf = bufs[:b] + (bufs[b][:w] + (n,) + bufs[b][w + 1:],) + bufs[b + 1:]
            elif act == 3:
                nb = arrive(bars, h.full(n), WARPS)
            elif w == 0:                             # act 4
                if not passes(bars, h.full(n), h.full_parity(n)):
                    continue
                if bufs[h.buffer(n)] != (n,) * WARPS:
                    return f"step {n} goes out with parts of {bufs[h.buffer(n)]}"
                nr, ni = reading + (n,), issued + 1
            pc = (n, act + 1) if act < 4 else (n + 1, 0)
            after.append((pcs[:w] + (pc,) + pcs[w + 1:], nb, nf, nr, ni))
        if not after and issued < STEPS:
            return f"nobody can go on: {pcs}"
        if not after and any(n < STEPS for n, _ in pcs):
            return f"a warp waits for good: {pcs}"
        for s in after:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


def test_every_order_of_the_warps(handover):
    assert explore(handover) is None


def test_the_model_sees_the_fault_of_one_barrier():
    assert explore(ONE_BARRIER).startswith("step 0 goes out with parts of")
