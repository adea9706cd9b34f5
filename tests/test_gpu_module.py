"""The autograd wrapper: forward and both gradients of NVFP4Linear against the oracle, and the per-call seed."""
import numpy as np
import pytest
import torch

from oracle import nvfp4_oracle as orc
from paper_2510_27527_b200 import synth
from tests.gpu_util import bf16_ulp_close, to_dev_bf16

pytestmark = pytest.mark.gpu


def test_module_forward_backward_match_the_oracle():
    from paper_2510_27527_b200 import binding as b
    from paper_2510_27527_b200.module import NVFP4Linear, call_seed

    N_tok, D, C = 192, 256, 128
    X, W, dY, ch = synth.layer_inputs(3, N_tok, D, C, n_outlier=3, factor=30.0, grad_scale=1e-3)
    lin = NVFP4Linear(D, C, cfg=b.LayerConfig(gs_mode=b.GS_TENSOR, seed=40, outliers=ch, rht=True))
    with torch.no_grad():
        lin.weight.copy_(to_dev_bf16(W))
    for call in range(2):  # every call has its own key, derived from the base seed, the module instance and the call number
        x = to_dev_bf16(X).reshape(4, 48, D).requires_grad_(True)
        y = lin(x)
        y.backward(to_dev_bf16(dY).reshape(4, 48, C))
        torch.cuda.synchronize()
        ocfg = orc.LayerConfig(gs_mode=orc.GS_TENSOR, seed=call_seed(40, lin.layer_id, call), outliers=ch, rht=True)
        Yo, so = orc.linear_fwd(X, W, ocfg)
        dXo, dWo = orc.linear_bwd_dx(dY, so, ocfg), orc.linear_bwd_dw(dY, so, ocfg)
        assert np.all(bf16_ulp_close(y.detach().reshape(N_tok, C).float().cpu().numpy(), Yo, 1.0, 1e-4 * np.abs(Yo).mean()))
        assert np.all(bf16_ulp_close(x.grad.reshape(N_tok, D).float().cpu().numpy(), dXo, 1.0, 1e-4 * np.abs(dXo).mean()))
        assert np.all(bf16_ulp_close(lin.weight.grad.float().cpu().numpy(), dWo, 1.0, 1e-4 * np.abs(dWo).mean()))
        lin.weight.grad = None


@pytest.mark.parametrize("tokens", [1, 77, 300])  # one saved buffer per call: its pieces at ragged sizes
@pytest.mark.parametrize("gs_mode,n_out", [(0, 0), (1, 0), (2, 5)])
def test_module_matches_the_binding_on_every_stream_and_thread(tokens, gs_mode, n_out):
    """The same calls through nvfp4_linear_fwd / nvfp4_linear_bwd with a buffer per array, and the module's on two streams from
    two threads at once: identical bytes everywhere."""
    import threading

    from paper_2510_27527_b200 import binding as b
    from paper_2510_27527_b200.module import NVFP4Linear, call_seed

    D, C = 200, 136
    X, W, dY, _ = synth.layer_inputs(3, tokens, D, C, n_outlier=3, factor=30.0, grad_scale=1e-3)
    outl = synth.outlier_channels(D, n_out, 5) if n_out else None
    x, w, dy = to_dev_bf16(X), to_dev_bf16(W), to_dev_bf16(dY)
    want = []
    for call in range(3):
        cfg = b.LayerConfig(gs_mode=gs_mode, seed=call_seed(7, 3, call), outliers=outl, dw_dtype=b.DT_BF16)
        y, saved = b.nvfp4_linear_fwd(x, w, cfg)
        want.append((y, *b.nvfp4_linear_bwd(dy, saved, cfg)))
    torch.cuda.synchronize()
    got, errors = {}, []

    def work(name):
        try:
            layer = NVFP4Linear(D, C, cfg=b.LayerConfig(gs_mode=gs_mode, seed=7, outliers=outl))
            layer.layer_id = 3
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                with torch.no_grad():
                    layer.weight.copy_(w)
                xi = x.clone().requires_grad_(True)
                out = []
                for _ in range(3):
                    y = layer(xi)
                    out.append((y, *torch.autograd.grad(y, (xi, layer.weight), dy)))
            s.synchronize()
            got[name] = out
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i in range(2):
        for a, bb in zip(got[i], want):
            for g, r in zip(a, bb):
                assert torch.equal(g, r)


def test_index_arrays_follow_the_outlier_channels():
    from paper_2510_27527_b200 import binding as b

    cfg = b.LayerConfig(outliers=np.array([1, 5]))
    first = cfg.index(16)
    assert cfg.index(16) is first
    cfg.outliers[1] = 7  # the same array with other contents
    outl, keep, cmap = cfg.index(16)
    assert outl.tolist() == [1, 7] and 5 in keep.tolist() and cmap.tolist()[5] == 4
    assert cfg.index(24)[1].numel() == 22


def test_layers_of_two_widths_share_a_configuration():
    """A module's call between a forward call and its separate backward calls changes nothing for them."""
    from paper_2510_27527_b200 import binding as b
    from paper_2510_27527_b200.module import NVFP4Linear

    mk = lambda r, c: torch.randn(r, c, device="cuda").to(torch.bfloat16)
    outl = [3, 40, 41, 199]
    x, w, dy, wide = mk(96, 200), mk(72, 200), mk(96, 72), mk(50, 1024)
    want_cfg = b.LayerConfig(seed=5, outliers=outl)
    _, saved = b.nvfp4_linear_fwd(x, w, want_cfg)
    want = b.nvfp4_linear_bwd(dy, saved, want_cfg)
    cfg = b.LayerConfig(seed=5, outliers=outl)
    layer = NVFP4Linear(1024, 64, cfg=cfg)
    _, saved = b.nvfp4_linear_fwd(x, w, cfg)
    with torch.no_grad():
        layer(wide)
    b.nvfp4_linear_fwd(wide, layer.weight.detach(), cfg)  # (and a direct call of that width)
    got = b.nvfp4_linear_bwd_dx(dy, saved, cfg), b.nvfp4_linear_bwd_dw(dy, saved, cfg)
    both = b.nvfp4_linear_bwd(dy, saved, cfg)
    for a, c, r in zip(got, both, want):
        assert torch.equal(a, r) and torch.equal(c, r)


def test_index_arrays_outlive_their_readers_on_other_streams():
    """Arrays uploaded on one stream, read by a call that another stream has yet to run, replaced meanwhile: their memory is not
    given to anyone before that call is done."""
    from paper_2510_27527_b200 import binding as b
    from paper_2510_27527_b200.module import NVFP4Linear

    D, outl = 4096, list(range(0, 4096, 13))
    layer = NVFP4Linear(D, 64, cfg=b.LayerConfig(outliers=outl))
    x = torch.randn(64, D, device="cuda").to(torch.bfloat16)
    side = torch.cuda.Stream()
    with torch.no_grad():
        want = layer(x)  # uploads on the current stream
        layer._calls = 0
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(100_000_000)  # (about 50 ms; the call below waits behind it)
            got = layer(x)
        layer.cfg._arrays._of.clear()
        ids = [torch.arange(n, dtype=torch.int32, device="cuda") for n in (len(outl), D - len(outl), D) for _ in range(8)]  # valid indexes, other ones
    torch.cuda.synchronize()
    assert torch.equal(got, want) and len(ids) == 24


@pytest.mark.filterwarnings("ignore::torch.jit.TracerWarning", "ignore::DeprecationWarning")
@pytest.mark.parametrize("grad", [False, True])
@pytest.mark.parametrize("weight_grad", [False, True])
def test_traces_and_tangents_do_not_pass_the_autograd_function_by(grad, weight_grad):
    import torch.autograd.forward_ad as fa

    from paper_2510_27527_b200.module import NVFP4Linear

    layer = NVFP4Linear(256, 136).requires_grad_(weight_grad)
    x = torch.randn(64, 256, device="cuda").to(torch.bfloat16)
    with torch.set_grad_enabled(grad):
        traced = torch.jit.trace(layer, x, check_trace=False)  # a recorded call keeps the key it was recorded with
        layer._calls = 0
        want = layer(2 * x)
        assert torch.equal(traced(2 * x), want)
        with fa.dual_level(), pytest.raises(NotImplementedError, match="jvp"):
            layer(fa.make_dual(x, torch.ones_like(x)))
        with fa.dual_level(), pytest.raises(NotImplementedError, match="jvp"):
            torch.func.functional_call(layer, {"weight": fa.make_dual(layer.weight.detach(), torch.ones_like(layer.weight))}, (x,))
