"""The router's layers at the edges of what its block reads ahead: hidden units below, at and above one round of the warps (64), and
of a lane's two weights of the second layer; inputs below and above what a lane holds at a time (32 x 7)."""
import pytest

from paper_2604_22808_b200 import configs as C

from test_parity_gpu import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,head_dim,t_embed_dim", [(1, 32, 2), (37, 32, 64), (64, 32, 128), (65, 64, 34), (130, 128, 70)])
def test_hidden_layer(hidden, head_dim, t_embed_dim):
    _run(C.TINY.scaled("hidden", router_hidden=hidden, head_dim=head_dim, t_embed_dim=t_embed_dim, heads=3))


# (units beyond the first 64 with just one load of eight inputs a lane, one input less, and with one behind what is held; an
# embedding as wide as the block and wider)
@pytest.mark.parametrize("hidden,head_dim,t_embed_dim", [(70, 64, 64), (70, 64, 62), (66, 32, 384), (66, 32, 386), (96, 32, 1024), (33, 32, 1040)])
def test_inputs_behind_those_held(hidden, head_dim, t_embed_dim):
    _run(C.TINY.scaled("inputs", router_hidden=hidden, head_dim=head_dim, t_embed_dim=t_embed_dim, heads=3))
