"""NVFP4Linear through its native autograd node against the same calls through the binding: identical bytes, and the same refusals."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def mk(*shape):
    return torch.randn(*shape, device="cuda").to(torch.bfloat16)


def run(layer, x, dy, native, monkeypatch, times=1):
    from paper_2510_27527_b200 import module as m

    with monkeypatch.context() as mp:
        if not native:
            mp.setattr(m, "_plain", lambda *a: False)
        layer._calls = 0
        x = x.clone().requires_grad_()
        y = layer(x)
        assert (y.grad_fn.name() == "NVFP4LinearBackward") == (native and y.dim() == 2 and layer.bias is None)
        out = [y.detach().clone()]
        for i in range(times):
            out += torch.autograd.grad(y, (x, *layer.parameters()), dy, retain_graph=i + 1 < times)
        with torch.no_grad():
            layer._calls = 0
            out.append(layer(x))
        assert not out[-1].requires_grad
        return out


@pytest.mark.parametrize("shape,D,C", [((1,), 256, 64), ((77,), 200, 136), ((3, 50), 136, 72)])
@pytest.mark.parametrize("opts", [dict(), dict(gs_mode=1), dict(gs_mode=2, rht=True, outliers=np.array([3, 40, 100])), dict(w_block16=True),
                                  dict(outliers=np.array([0, 7]), outlier_fp8=True, concurrent=False)])
def test_same_bytes_as_through_the_binding(shape, D, C, opts, monkeypatch):
    from paper_2510_27527_b200 import binding as b
    from paper_2510_27527_b200.module import NVFP4Linear

    layer = NVFP4Linear(D, C, bias=len(shape) == 2, cfg=b.LayerConfig(seed=11, **opts))
    layer.layer_id = 0
    x = mk(*shape, D)
    wide = mk(*shape, 2 * C)
    for dy in (wide[..., :C], mk(*shape, C), mk(1).expand(*shape, C)):
        for times in (1, 2):  # twice over the same call
            got, want = (run(layer, x, dy, native, monkeypatch, times) for native in (True, False))
            assert len(got) == len(want) and all(torch.equal(a, r) and a.stride() == r.stride() for a, r in zip(got, want))


@pytest.mark.parametrize("rounding", [(0, 0, 1), (), (0, 0, 2, 1, 1)])
def test_roundings_that_are_not_given_are_to_nearest(rounding, monkeypatch):
    from paper_2510_27527_b200 import binding as b
    from paper_2510_27527_b200.module import NVFP4Linear

    layer = NVFP4Linear(256, 64, cfg=b.LayerConfig(seed=11, rounding=rounding))
    layer.layer_id = 0
    x, dy = mk(96, 256), mk(96, 64)
    got, want = (run(layer, x, dy, native, monkeypatch) for native in (True, False))
    layer.cfg.rounding = (*rounding, 0, 0, 0, 0, 0, 0)[:6]
    assert all(torch.equal(a, r) and torch.equal(a, f) for a, r, f in zip(got, want, run(layer, x, dy, True, monkeypatch)))


def test_rows_of_an_odd_width_are_padded(monkeypatch):
    from paper_2510_27527_b200 import module as m

    layer = m.NVFP4Linear(200, 133)
    x = mk(77, 200)
    got = []
    for native in (True, False):
        with monkeypatch.context() as mp, torch.no_grad():
            if not native:
                mp.setattr(m, "_plain", lambda *a: False)
            layer._calls = 0
            got.append(layer(x))
    assert torch.equal(*got) and got[0].stride() == got[1].stride() == (136, 1) and got[0].untyped_storage().nbytes() == 77 * 136 * 2


def test_under_capture_and_from_a_changed_configuration(monkeypatch):
    from paper_2510_27527_b200 import binding as b
    from paper_2510_27527_b200.module import NVFP4Linear

    layer = NVFP4Linear(256, 128, cfg=b.LayerConfig(gs_mode=b.GS_TENSOR, seed=3))
    layer.layer_id = 0
    x, dy = mk(96, 256), mk(96, 128)
    want = run(layer, x, dy, False, monkeypatch)
    layer._calls = 0
    xi = x.clone().requires_grad_()
    torch.autograd.grad(layer(xi), (xi, layer.weight), dy)  # (torch's engine starts its threads)
    layer._calls = 0
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        y = layer(xi)
        layer.cfg.gs_mode = b.GS_ROW  # belongs to later calls
        grads = torch.autograd.grad(y, (xi, layer.weight), dy)
    layer.cfg.gs_mode = b.GS_TENSOR
    graph.replay()
    torch.cuda.synchronize()
    for a, r in zip((y, *grads), want):
        assert torch.equal(a, r)


def test_errors_are_the_bindings():
    from paper_2510_27527_b200 import binding as b
    from paper_2510_27527_b200.module import NVFP4Linear

    layer = NVFP4Linear(64, 64, cfg=b.LayerConfig(gs_mode=7))
    with pytest.raises(b.Nvfp4Error, match="nvfp4_linear_fwd"), torch.no_grad():
        layer(mk(16, 64))
    layer = NVFP4Linear(64, 64, cfg=b.LayerConfig(gs_mode=b.GS_BLOCK128))
    x = mk(16384 + 128, 64).requires_grad_()  # the weight gradient's K is beyond what outer-block products take
    y = layer(x)
    with pytest.raises(b.Nvfp4Error, match="nvfp4_linear_bwd"):
        y.sum().backward()
    with pytest.raises(RuntimeError, match="input on cpu"):
        layer(torch.zeros(4, 64, dtype=torch.bfloat16))
