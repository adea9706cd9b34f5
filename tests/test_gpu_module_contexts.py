"""NVFP4Linear where its native autograd node does not serve: under compilation, with weights and inputs that are not plain tensors and
parameters. The bytes are those of an ordinary call."""
import pytest
import torch

pytestmark = pytest.mark.gpu

T, D, C = 96, 256, 128


def mk(*shape):
    return torch.randn(*shape, device="cuda").to(torch.bfloat16)


def layer(w, **opts):
    from paper_2510_27527_b200 import binding as b
    from paper_2510_27527_b200.module import NVFP4Linear

    made = NVFP4Linear(D, C, cfg=b.LayerConfig(seed=3, **opts))
    made.layer_id = 0
    with torch.no_grad():
        made.weight.copy_(w)
    return made


@pytest.fixture
def data():
    """(x, w, dy, what an ordinary step of a layer with these gives)."""
    x, w, dy = mk(T, D), mk(C, D), mk(T, C)
    plain, xi = layer(w), x.clone().requires_grad_()
    y = plain(xi)
    return x, w, dy, (y.detach(), *torch.autograd.grad(y, (xi, plain.weight), dy))


def same(got, want):
    return all(torch.equal(g.detach().as_subclass(torch.Tensor), r) for g, r in zip(got, want))


@pytest.mark.parametrize("backend", ["eager", "inductor"])
@pytest.mark.parametrize("warm", [False, True])  # whether the thread has its second stream already
def test_compiled(data, backend, warm):
    from paper_2510_27527_b200 import binding as b

    x, w, dy, want = data
    torch._dynamo.reset()
    b._thread.__dict__.clear()
    if warm:
        b.thread_side(x.device, b._stream_ptr())
    with torch.no_grad():
        assert same((torch.compile(layer(w), backend=backend)(x),), want)
    made, xi = layer(w), x.clone().requires_grad_()
    y = torch.compile(made, backend=backend)(xi)
    assert same((y, *torch.autograd.grad(y, (xi, made.weight), dy)), want)
    torch._dynamo.reset()
