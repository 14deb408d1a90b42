"""Routers wider than the shared memory a block has by default, and one wider than it can have: the layer runs under a given
allocation all the same."""
import os
import subprocess
import sys

import pytest

from paper_2604_22808_b200 import configs as C
from paper_2604_22808_b200 import inputs as I

from test_parity_gpu import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t_embed_dim", [9800, 11800, 50000])
def test_wide_timestep_embedding(t_embed_dim):
    _run(C.TINY.scaled("wide", t_embed_dim=t_embed_dim))


def test_wider_than_shared_memory():
    import torch
    from paper_2604_22808_b200 import binding as B
    cfg = C.TINY.scaled("widest", t_embed_dim=60000)
    _run(cfg, alloc=[7, 2])
    plan = B.Plan(cfg, I.router_weights(cfg))
    x = torch.zeros(plan._shape, device="cuda")
    with pytest.raises(B.FFError) as e:
        plan.forward(x, x, x, torch.empty_like(x), timesteps=[500.0])
    assert e.value.status == 4
    plan.destroy()


EDGES = r"""
import sys
sys.path.insert(0, %r); sys.path.insert(0, %r)
from paper_2604_22808_b200 import configs as C
from test_parity_gpu import _run
for n in (9944, 9946, 10000, 10072, 10080, 10082):
    _run(C.TINY.scaled("edge", t_embed_dim=n))
    print("ran", n)
"""


def test_around_the_default_shared_memory():
    """8192 + 4 (3 x 32 + t_embed_dim + 64) bytes of dynamic shared memory, from 544 below the 48 KB that a launch has without asking
    to just above them: what the kernel declares statically counts, too.  In a process of its own: what a
    wider router has asked for stays with the kernel."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", EDGES % (root, os.path.join(root, "tests"))], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split("\n")[-2] == "ran 10082", r.stdout[-500:] + r.stderr[-2000:]


def test_a_narrower_plan_made_later():
    import torch
    from paper_2604_22808_b200 import binding as B
    wide, narrow = (C.TINY.scaled("width", t_embed_dim=n) for n in (50000, 11800))
    first = B.Plan(wide, I.router_weights(wide))
    x = torch.randn(first._shape, device="cuda")
    out, again = torch.empty_like(x), torch.empty_like(x)
    first.forward(x, x, x, out, timesteps=[500.0])
    second = B.Plan(narrow, I.router_weights(narrow))
    first.forward(x, x, x, again, timesteps=[500.0])
    second.forward(x, x, x, torch.empty_like(x), timesteps=[500.0])
    assert first.device_status() == 0 and second.device_status() == 0 and torch.equal(out, again)
    first.destroy(); second.destroy()
