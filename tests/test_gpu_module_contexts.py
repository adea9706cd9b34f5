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


@pytest.mark.parametrize("backend", ["eager", "inductor"])
@pytest.mark.parametrize("opts", [dict(), dict(gs_mode=2, rht=True, outliers=[3, 40, 100]), dict(concurrent=False)])
def test_compiled_autograd_over_ordinary_calls(opts, backend):
    """A recorded backward, run again on later calls with other keys, inputs and weights: each has its own draws and saved operands."""
    from torch._dynamo import compiled_autograd

    first, second = mk(D, D), mk(C, D)
    torch._dynamo.reset()
    for step in range(3):
        x, dy = mk(T + 8 * (step == 2), D), mk(T + 8 * (step == 2), C)
        got = []
        for compiled in (False, True):
            from paper_2510_27527_b200 import binding as b
            from paper_2510_27527_b200.module import NVFP4Linear

            model = torch.nn.Sequential(NVFP4Linear(D, D, cfg=b.LayerConfig(seed=3, **opts)), torch.nn.ReLU(), layer(second, **opts))
            model[0].layer_id = 1
            with torch.no_grad():
                model[0].weight.copy_(first)
            for m in (model[0], model[2]):
                m._calls = step
            xi = x.clone().requires_grad_(step > 0)
            y = model(xi)
            if compiled:
                with compiled_autograd._enable(torch.compile(backend=backend)):
                    y.backward(dy)
            else:
                y.backward(dy)
            got.append((y.detach(), model[0].weight.grad, model[2].weight.grad, *([xi.grad] if step else [])))
        assert same(*got)
    torch._dynamo.reset()


def test_compiled_autograd_over_an_excluded_layer(data):
    import torch._dynamo.config

    x, w, dy, want = data
    torch._dynamo.reset()
    made, xi = layer(w), x.clone().requires_grad_()
    apart = torch.compiler.disable(made)

    @torch.compile(backend="eager")
    def step(xi):
        y = apart(xi)
        y.backward(dy)
        return y

    with torch._dynamo.config.patch(compiled_autograd=True):
        assert same((step(xi), xi.grad, made.weight.grad), want)
    torch._dynamo.reset()


class Marked(torch.Tensor):
    pass


@pytest.mark.parametrize("which", ["weight", "input"])
def test_calls_without_gradients_pass_the_autograd_function_by(data, which, monkeypatch):
    from paper_2510_27527_b200 import module

    x, w, _, want = data
    monkeypatch.setattr(module._NVFP4LinearFn, "apply", lambda *a: pytest.fail("autograd function"))
    with torch.no_grad():
        y = torch.func.functional_call(layer(w), {"weight": w}, (x,)) if which == "weight" else layer(w)(x.as_subclass(Marked))
    assert same((y,), want)
    y = torch.func.functional_call(layer(w), {"weight": w}, (x,))  # with gradients on, but none asked for
    assert same((y,), want) and not y.requires_grad


@pytest.mark.parametrize("grad", [False, True])
def test_transforms_are_refused(data, grad):
    x, w, _, _ = data
    with torch.set_grad_enabled(grad):
        for call in (lambda m: torch.func.grad(lambda t: m(t).float().sum())(x), lambda m: torch.func.vmap(m)(x[None])):
            with pytest.raises(RuntimeError, match="setup_context"):
                call(layer(w))


def test_other_weights_and_inputs_with_gradients(data):
    import torch.nn.utils.parametrize as parametrize

    class Same(torch.nn.Module):
        def forward(self, w):
            return w * 1

    x, w, dy, want = data
    xi, wi = x.clone().requires_grad_(), w.clone().requires_grad_()
    y = torch.func.functional_call(layer(w), {"weight": wi}, (xi,))
    assert same((y, *torch.autograd.grad(y, (xi, wi), dy)), want)
    made = layer(w)
    parametrize.register_parametrization(made, "weight", Same())
    y = made(xi)
    assert same((y, *torch.autograd.grad(y, (xi, made.parametrizations.weight.original), dy)), want)
    made, xi = layer(w), x.clone().as_subclass(Marked).requires_grad_()
    y = made(xi)
    y.backward(dy)
    assert same((y, xi.grad, made.weight.grad), want)


def test_the_node_called_by_hand(data):
    x, w, dy, want = data
    y = layer(w)(x.clone().requires_grad_())
    assert same((y, *y.grad_fn(dy)), want)
    assert same((y, *y.grad_fn(dy.float())), want)
    for bad in (dy[:-1], dy[:, :-1], dy[0], dy[None], mk(T + 1, C), dy.cpu(), mk(C, T)):
        with pytest.raises(RuntimeError, match=r"gradient of shape .* for an output of shape \[96, 128\]"):
            y.grad_fn(bad)
    assert same((y, *y.grad_fn(dy)), want)


@pytest.mark.parametrize("opts", [dict(), dict(outliers=[3, 40, 100])])
def test_what_backward_reads_on_another_stream_outlives_it(data, opts):
    """The node called on a stream that has yet to get there, and dropped meanwhile: its buffer is not given to anyone before that."""
    x, w, dy, _ = data
    made = layer(w, **opts)
    xi = x.clone().requires_grad_()
    made(xi).backward(dy)
    want = (xi.grad, made.weight.grad)
    made._calls = 0
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    y = made(xi)
    held = torch.cuda.memory_allocated() - before - y.untyped_storage().nbytes()  # the buffer, as the allocator rounds it
    other = torch.cuda.Stream()
    other.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(other):
        torch.cuda._sleep(100_000_000)  # (about 50 ms)
        got = y.grad_fn(dy)
    del y
    pending = sum(block["size"] for s in torch.cuda.memory_snapshot() for block in s["blocks"] if block["state"] == "active_pending_free")
    filled = [torch.zeros(n, dtype=torch.uint8, device="cuda") for n in (held,) * 8]
    torch.cuda.synchronize()
    assert held > 0 and pending >= held and len(filled) == 8 and same(got, want)


def test_what_the_node_holds_is_no_saved_variable(data):
    """As with the autograd function: hooks see nothing of it, and a second backward runs."""
    x, w, dy, want = data
    made, xi, seen = layer(w), x.clone().requires_grad_(), []
    with torch.autograd.graph.saved_tensors_hooks(lambda t: seen.append(t) or t, lambda t: t):
        y = made(xi)
    for _ in range(2):
        xi.grad = made.weight.grad = None
        y.backward(dy)
        assert same((y, xi.grad, made.weight.grad), want)
    assert seen == []
