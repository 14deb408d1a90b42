"""Routers wider than the shared memory a block has by default, and one wider than it can have: the layer runs under a given
allocation all the same."""
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
