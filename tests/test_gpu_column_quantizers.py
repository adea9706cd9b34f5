"""The column-axis quantizers that transpose in registers, at the edges of their tiles, against the oracle: exact."""
import numpy as np
import pytest

from oracle import nvfp4_oracle as orc
from paper_2510_27527_b200 import synth
from tests.gpu_util import assert_operand_equal, to_dev_bf16

pytestmark = pytest.mark.gpu

# (source rows = operand k, source columns = operand rows): one row; one below, at and above an inner block, an outer block of 128 and
# a second one; fewer columns than a lane group, one group less and more than a CTA's 64, columns past a 128-row scale tile
SHAPES = [(1, 4), (15, 12), (16, 60), (17, 64), (127, 68), (128, 16), (129, 132), (255, 20), (257, 260)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("gs_mode", [orc.GS_TENSOR, orc.GS_ROW, orc.GS_BLOCK128])
@pytest.mark.parametrize("rounding", [orc.RTN, orc.SR, orc.SR_SCALE_UP])
@pytest.mark.parametrize("rht", [0, 9])
def test_edges(shape, gs_mode, rounding, rht):
    from paper_2510_27527_b200 import binding as b

    x = synth.gradients(shape[0], shape[1], 3 + shape[0], 1e-3)
    x[-1, -1] = 0.5  # the maximum in the last element
    x = synth.round_to_bf16(x)
    xt = np.ascontiguousarray(x.T)
    ref = orc.quantize(orc.rht16(xt, 42, rht) if rht else xt, orc.AXIS_ROW, rounding, gs_mode, seed=42, stream_id=5)
    for layout in (b.SF_TILED128x4, b.SF_LINEAR):
        out = b.alloc_operand(shape[1], shape[0], gs_mode, layout, poison=True)
        src = to_dev_bf16(np.pad(x, ((0, 0), (0, -shape[1] % 8))))[:, : shape[1]]
        b.nvfp4_quantize(src, b.AXIS_COL, rounding, 42, 5, gs_mode, layout, out=out, rht_stream_id=rht)
        assert_operand_equal(out, ref, f"{shape} gs{gs_mode} r{rounding} rht{rht} layout{layout}", k_extended=rht != 0)


# the largest grid of 128 x 64 tiles that runs three CTAs per SM (592 on 148 SMs), the next one, and a ragged one
@pytest.mark.parametrize("shape", [(4736, 1024), (4740, 1024), (4999, 1000)])
@pytest.mark.parametrize("rht", [0, 9])
def test_requantize_outer_block_large(shape, rht):
    from paper_2510_27527_b200 import binding as b

    x, _ = synth.activations(shape[0], shape[1], 11, n_outlier=3, factor=50.0)
    fwd_ref = orc.quantize(x, orc.AXIS_ROW, orc.RTN, orc.GS_BLOCK128)
    xt = np.ascontiguousarray(orc.rematerialize_f32(fwd_ref).T)
    ref = orc.quantize(orc.rht16(xt, 5, rht) if rht else xt, orc.AXIS_ROW, orc.SR, orc.GS_BLOCK128, seed=5, stream_id=6)
    fwd = b.nvfp4_quantize(to_dev_bf16(x), b.AXIS_ROW, b.ROUND_RTN, 0, 1, b.GS_BLOCK128)
    out = b.alloc_operand(shape[1], shape[0], b.GS_BLOCK128, poison=True)
    b.nvfp4_requantize_t(fwd, b.ROUND_SR, 5, 6, out=out, rht_stream_id=rht)
    assert_operand_equal(out, ref, f"{shape} rht{rht}", k_extended=rht != 0)
