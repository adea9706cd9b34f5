"""GPU parity of stochastic rounding where its cells change: values on the grid points, on cell boundaries and next to them, either
side of 1 (where the spacing of the grid changes), at and above 6, zeros of both signs and subnormals; under block scales of every
size down to the subnormal ones, under which a block's largest values lie up to half again beyond the grid's end."""
import numpy as np
import pytest

from oracle import nvfp4_oracle as orc
from tests.gpu_util import assert_operand_equal, to_dev_bf16

pytestmark = pytest.mark.gpu


def edge_values(rows, cols, seed):
    """[rows, cols] BF16-representable values: blocks of 16 along a row, the j-th at scale 2^-(j % 14), or 1.4 times that (a block
    scale that has to be rounded); the tensor's maximum is 2688, so that its global scale is 1."""
    rng = np.random.default_rng(seed)
    grid = np.array([0, 0.5, 1, 1.5, 2, 3, 4, 6])
    near = np.concatenate([grid, grid * (1 + 2.0 ** -7), grid * (1 - 2.0 ** -8), 0.5 * (grid[1:] + grid[:-1]), [2.0 ** -8, 2.0 ** -20, 0.25, 0.75]])
    x = rng.choice(near, (rows, cols)) * rng.choice([-1.0, 1.0], (rows, cols))
    x = np.where(rng.random((rows, cols)) < 0.3, x * (1 + rng.random((rows, cols)) * 0.2), x)
    j = np.arange(cols) // 16
    x = x * 2.0 ** -(j % 14) * np.where(j % 3 == 2, 1.4, 1.0)
    x[:, 5::97] = -0.0
    x[:, 3::89] = 2.0 ** -130
    x[rows // 2, 1] = 2688.0
    bits = np.ascontiguousarray(x, dtype=np.float32).view(np.uint32) & np.uint32(0xFFFF0000)
    return bits.view(np.float32)


@pytest.mark.parametrize("rows,cols", [(16, 256), (130, 896), (33, 2000)])
@pytest.mark.parametrize("gs_mode", [orc.GS_TENSOR, orc.GS_ROW, orc.GS_BLOCK128])
@pytest.mark.parametrize("axis", [orc.AXIS_ROW, orc.AXIS_COL])
def test_stochastic_rounding_at_cell_edges(rows, cols, gs_mode, axis):
    from paper_2510_27527_b200 import binding as b

    x = edge_values(rows, cols, rows + gs_mode)
    if axis == orc.AXIS_COL:  # the blocks run down the columns
        x = np.ascontiguousarray(np.pad(x, ((0, -rows % 8), (0, 0))).T)
    for seed in (0, 0xFEDCBA9876543210):
        ref = orc.quantize(x, axis, orc.SR, gs_mode, seed=seed, stream_id=5)
        R, K = (x.shape[0], x.shape[1]) if axis == orc.AXIS_ROW else (x.shape[1], x.shape[0])
        out = b.alloc_operand(R, K, gs_mode, poison=True)
        b.nvfp4_quantize(to_dev_bf16(x), axis, b.ROUND_SR, seed, 5, gs_mode, out=out)
        assert_operand_equal(out, ref, f"{rows}x{cols} gs{gs_mode} axis{axis} seed{seed}")
