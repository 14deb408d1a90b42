"""The binding's own checks, on the CPU: what may stand for the timesteps, that nothing shorter than what the library
reads reaches it, and where the stream handle comes from."""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

from paper_2604_22808_b200 import binding as B
from paper_2604_22808_b200 import configs as C


@pytest.mark.parametrize("values", [800.0, 800, np.float32(800), np.array(800.0), [800.0], (800,), np.array([800.0]), np.array([[800.0]]),
                                    [[800.0]], torch.tensor([800.0]), torch.tensor(800.0), range(800, 801)], ids=repr)
def test_one_sample(values):
    assert list(B._floats(values, 1)) == [800.0]


def test_several_samples():
    assert B._floats(None, 2) is None
    assert list(B._floats([1, 2.5], 2)) == [1.0, 2.5]
    assert list(B._floats(np.array([[1.0], [2.5]]), 2)) == [1.0, 2.5]
    assert list(B._floats([1, 2, 3], 2)) == [1.0, 2.0, 3.0]       # (the library reads the first two)
    for short in (1.0, [1.0], [], np.zeros(1)):
        with pytest.raises(B.FFError) as e:
            B._floats(short, 2)
        assert e.value.status == 1 and "timesteps" in str(e.value)


@pytest.fixture
def plan():
    """A plan without a handle: the library refuses it, so a message of the binding shows who refused."""
    p = object.__new__(B.Plan)
    p.cfg = C.TINY.scaled("two", batch=2)
    p._torch, p.device, p.handle = torch, torch.device("cpu"), None
    p._shape = torch.Size((2, C.TINY.heads, C.TINY.T, C.TINY.H, C.TINY.W, C.TINY.head_dim))
    p._dtype = torch.float32
    p._stream = lambda: None
    return p


def test_short_arguments_are_refused(plan):
    x = torch.zeros(plan._shape)
    n = 2 * C.TINY.heads
    masks = torch.zeros(n, dtype=torch.uint8)
    bad_masks = (masks[:-1], torch.zeros(n, dtype=torch.int32), torch.zeros(2 * n, dtype=torch.uint8)[::2], masks.to("meta"))
    for call in (plan.forward, lambda q, k, v, o, **kw: plan.route(q, k, v, kw["timesteps"], kw.get("alloc"))):
        with pytest.raises(B.FFError, match="timesteps"):
            call(x, x, x, x, timesteps=[1.0])
        for m in bad_masks:
            with pytest.raises(B.FFError, match="band masks"):
                call(x, x, x, x, timesteps=[1.0, 2.0], alloc=m)
        with pytest.raises(B.FFError, match="plan is NULL"):
            call(x, x, x, x, timesteps=[1.0, 2.0], alloc=masks)
    with pytest.raises(B.FFError, match="timesteps"):
        plan.forward_host(x, x, x, x, timesteps=1.0)
    with pytest.raises(B.FFError, match="band masks"):
        plan.forward_host(x, x, x, x, alloc_host=np.zeros(n - 1, np.uint8))
    for i in range(4):
        for wrong in (x[:1], x.half(), x.transpose(0, 1)):
            args = [x, x, x, x]
            args[i] = wrong
            with pytest.raises(B.FFError, match="shape"):
                plan.forward_host(*args, timesteps=[1.0, 2.0])
    with pytest.raises(B.FFError, match="plan is NULL"):
        plan.forward_host(x, x, x, x, alloc_host=np.zeros(n, np.uint8))


def test_short_arguments_of_the_projected_layer(plan):
    plan.cfg = C.R64K.scaled("two", batch=2)
    D = plan.cfg.heads * plan.cfg.head_dim

    class Fake:                                                     # (the call wants CUDA tensors: only what it looks at)
        dtype, device, is_cuda = torch.bfloat16, plan.device, True

        def __init__(self, *shape):
            self.shape = shape

        def is_contiguous(self):
            return True

        def data_ptr(self):
            return 0

    x = Fake(2, plan.cfg.N, D)
    args = (x, Fake(3, D, D), Fake(D, D), x)
    with pytest.raises(B.FFError, match="timesteps"):
        plan.forward_projected(*args, timesteps=[1.0])
    with pytest.raises(B.FFError, match="band masks"):
        plan.forward_projected(*args, alloc=torch.zeros(1, dtype=torch.uint8))
    with pytest.raises(B.FFError, match="plan is NULL"):
        plan.forward_projected(*args, timesteps=[1.0, 2.0])


def test_stream_handle_with_and_without_the_private_name():
    public = SimpleNamespace(current_stream=lambda index: SimpleNamespace(cuda_stream=100 + index))
    assert B._stream_getter(SimpleNamespace(_C=SimpleNamespace(), cuda=public))(3) == 103
    private = SimpleNamespace(_cuda_getCurrentRawStream=lambda index: 200 + index)
    assert B._stream_getter(SimpleNamespace(_C=private, cuda=public))(3) == 203
