"""The compacting row quantizer (columns from a list): operand bytes against the oracle on the compacted matrix, and the BF16 side
operand that the same launch writes against plain indexing. Both are exact."""
import numpy as np
import pytest
import torch

from oracle import nvfp4_oracle as orc
from paper_2510_27527_b200 import synth
from tests.gpu_util import assert_operand_equal, to_dev_bf16, to_dev_i32

pytestmark = pytest.mark.gpu


def B():
    from paper_2510_27527_b200 import binding

    return binding


def _keep(cols, n_out):
    out = np.sort(np.random.default_rng(cols + n_out).choice(cols, n_out, replace=False)).astype(np.int32)
    return np.setdiff1d(np.arange(cols), out).astype(np.int32), out


# (rows, columns, columns left out): one row; fewer rows than a CTA takes, one more; one column kept; kept columns one below, at and
# one above a multiple of 128; the widest source that four rows of a CTA stage (3072 elements with the compact row), the next one;
# columns that are no multiple of 8; two rows at the limit of shared memory, and past it (element by element)
SHAPES = [(1, 16, 1), (3, 136, 9), (5, 136, 8), (4, 264, 263), (9, 136, 7), (129, 264, 1), (33, 1536, 5), (33, 1544, 5), (6, 100, 3), (3, 25600, 30),
          (3, 25736, 3)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("gs_mode", [orc.GS_TENSOR, orc.GS_ROW, orc.GS_BLOCK128])
@pytest.mark.parametrize("rounding", [orc.RTN, orc.SR])
def test_kept_columns(shape, gs_mode, rounding):
    b = B()
    rows, cols, n_out = shape
    keep, _ = _keep(cols, n_out)
    x, _ = synth.activations(rows, cols, 5 + cols, n_outlier=1, factor=50.0)
    ref = orc.quantize(np.ascontiguousarray(x[:, keep]), orc.AXIS_ROW, rounding, gs_mode, seed=77, stream_id=1)
    for layout in (b.SF_LINEAR, b.SF_TILED128x4):
        out = b.alloc_operand(rows, len(keep), gs_mode, layout, poison=True)
        src = to_dev_bf16(np.pad(x, ((0, 0), (0, -cols % 8))))[:, :cols]  # rows start on 16-byte boundaries
        b.nvfp4_quantize(src, b.AXIS_ROW, rounding, 77, 1, gs_mode, layout, keep_cols=to_dev_i32(keep), out=out)
        assert_operand_equal(out, ref, f"{shape} gs{gs_mode} r{rounding} layout{layout}")


@pytest.mark.parametrize("tokens,D,n_out", [(1, 64, 1), (3, 264, 65), (5, 1536, 64), (130, 1544, 63), (3, 25736, 2)])
@pytest.mark.parametrize("gs_mode", [orc.GS_TENSOR, orc.GS_ROW, orc.GS_BLOCK128])
def test_side_operand(tokens, D, n_out, gs_mode):
    b = B()
    if gs_mode == orc.GS_BLOCK128 and D > 16384:
        pytest.skip("wider than the product of this scale mode takes")
    _, out = _keep(D, n_out)
    g = torch.Generator(device="cuda").manual_seed(tokens + D)
    x = torch.randn(tokens, D, generator=g, device="cuda").bfloat16()
    w = torch.randn(72, D, generator=g, device="cuda").bfloat16()
    cfg = b.LayerConfig(gs_mode=gs_mode, seed=3, outliers=out)
    cfg.prepare(D)
    saved = b.alloc_saved(x, w, cfg)
    for side in (saved.X_out, saved.W_out):
        side.fill_(-7.0)
    b.nvfp4_linear_fwd(x, w, cfg, saved=saved)
    torch.cuda.synchronize()
    idx = torch.from_numpy(out).long().cuda()
    for side, src in ((saved.X_out, x), (saved.W_out, w)):
        assert torch.equal(side[:, :n_out], src[:, idx])
        assert not side[:, n_out:].any()
