"""Infinite inputs of the simulated FP6 layer's operands: a block whose scale is not a number is written as -0, by the row quantizer, by the
transposing re-quantizer and by the expansion of an FP4 operand; blocks of finite values beside it, under the same infinite global scale,
are written as zeros with their signs."""

import pytest
import torch

from paper_2510_27527_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rounding", [0, 1])
@pytest.mark.parametrize("bad", [float("inf"), -float("inf")])
def test_blocks_with_an_infinity_are_written_as_negative_zeros(rounding, bad):
    x = torch.randn(64, 256, device="cuda", dtype=torch.bfloat16)
    x[5, 33] = bad
    block = torch.zeros(64, 256, dtype=torch.bool, device="cuda")
    block[5, 32:48] = True
    for workspace in (16, 256):
        out = b.nvfp4_fp6_quantize(x, rounding, 7, 1, workspace=torch.zeros(workspace, dtype=torch.uint8, device="cuda"))
        assert out.gscale.isinf().all()
        bits = out.vals[:, :256].view(torch.int16)
        assert (bits[block] == -32768).all() and (out.vals[:, :256][~block] == 0).all()
    t = b.nvfp4_fp6_requantize_t(out, rounding, 7, 2)
    assert not t.vals.isnan().any()
    e = b.nvfp4_expand_operand(b.nvfp4_quantize(x))
    assert not e.vals.isnan().any() and (e.vals[:, :256].view(torch.int16)[block] == -32768).all()
