"""What NVFP4Linear refuses before it touches a device."""
import pytest
import torch


@pytest.mark.parametrize("grad", [False, True])
@pytest.mark.parametrize("shape", [(64, 128), (64, 512), (128,), (4, 16, 512), (2, 128), (0, 128), ()])
def test_inputs_of_another_width_are_refused(shape, grad):
    from paper_2510_27527_b200.module import NVFP4Linear

    layer = NVFP4Linear(256, 64, device="cpu")
    with torch.set_grad_enabled(grad), pytest.raises(RuntimeError, match="256 input features"):
        layer(torch.zeros(shape, dtype=torch.bfloat16))
    assert layer._calls == 0  # no key of the layer's sequence is used up


def _call(**opts):
    from paper_2510_27527_b200 import binding as b
    from paper_2510_27527_b200.module import NVFP4Linear

    NVFP4Linear(256, 64, device="cpu", cfg=b.LayerConfig(**opts))(torch.zeros(4, 256, dtype=torch.bfloat16))


def test_a_message_with_a_number_is_an_exception():
    with pytest.raises((TypeError, IndexError), match="has 7 entries"):  # (it ended the process where the node had a C++ library of its own)
        _call(rounding=(0, 0, 1, 1, 1, 1, 1))


@pytest.mark.parametrize("opts", [dict(rounding=(0, 0, 1)), dict(rounding=()), dict(rounding=[0, 0, True, 1, 1, 1]), dict(gs_mode=True), dict(rht="1"),
                                  dict(w_block16=1 << 70)])
def test_configurations_that_the_c_structure_takes_are_taken(opts):
    with pytest.raises(RuntimeError, match="input on cpu"):  # the first thing that is refused after the configuration
        _call(**opts)


@pytest.mark.parametrize("opts", [dict(gs_mode=1.0), dict(gs_mode="1"), dict(gs_mode=None), dict(rounding=(0, 0, 1.0, 1, 1, 1)), dict(rounding="001111"),
                                  dict(rounding=None), dict(rht=None), dict(rht="x")])
def test_configurations_that_the_c_structure_refuses_are_refused(opts):
    with pytest.raises((TypeError, ValueError)):
        _call(**opts)
