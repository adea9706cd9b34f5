"""The weights' backward operand of a layer with outlier channels: kept and outlier channels of it are quantized by one launch or, for other
roundings and large weights, by two. Every byte equals what the element-wise kernel of nvfp4_requantize_t with a row map gives, which reads
the forward operand and the BF16 weights column by column."""

import numpy as np
import pytest
import torch

from paper_2510_27527_b200 import binding as b

pytestmark = pytest.mark.gpu

# (C, D, outlier channels): one tile of each source; tiles of 64 channels and of 128 weight rows that end inside; one outlier channel; more
# outlier than kept channels; 3 and 4 x 148 CTAs of kept channels (the outer block's limit) and 32 x 148 (the others')
SIZES = [(16, 16, 8), (128, 128, 64), (136, 200, 1), (129, 192, 65), (1000, 264, 200), (2816, 1024, 102), (4736, 1024, 8), (4737, 1032, 8),
         (4097, 9480, 8)]


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("gs", [b.GS_TENSOR, b.GS_ROW, b.GS_BLOCK128])
@pytest.mark.parametrize("rounding", [b.ROUND_SR, b.ROUND_SR_SCALE_UP, b.ROUND_RTN])
def test_operand_equals_the_element_wise_kernel(size, gs, rounding):
    C, D, n_out = size
    rng = np.random.RandomState(C + D)
    outl = np.sort(rng.permutation(D)[:n_out]).astype(np.int32)
    gen = torch.Generator(device="cuda").manual_seed(C)
    draw = lambda *s: torch.randn(*s, generator=gen, device="cuda", dtype=torch.bfloat16)
    ld = (C + 7) // 8 * 8
    x, w, dy = draw(32, D), draw(C, D), draw(32, ld)[:, :C]
    w[:, torch.from_numpy(outl).cuda().long()] *= 40
    cfg = b.LayerConfig(gs_mode=gs, seed=11, outliers=outl, rounding=(b.ROUND_RTN, b.ROUND_RTN, b.ROUND_SR, rounding, b.ROUND_SR, b.ROUND_SR))
    _, saved = b.nvfp4_linear_fwd(x, w, cfg, Y=torch.empty(32, ld, device="cuda", dtype=torch.bfloat16)[:, :C])
    ws = b.linear_workspace(b.OP_BWD_DX, 32, D, C, cfg)
    ws.fill_(0xA5)
    b.nvfp4_linear_bwd_dx(dy, saved, cfg, workspace=ws)
    got = b.nvfp4_linear_bwd_operand(b.OP_BWD_DX, 4, 32, D, C, cfg, ws)
    cmap = np.full(D, -1, dtype=np.int32)
    cmap[np.setdiff1d(np.arange(D), outl)] = np.arange(D - n_out)
    want = b.alloc_operand(D, C, gs)
    b.nvfp4_requantize_t(saved.qw, rounding, 11, 4, hp=w, row_map=torch.from_numpy(cmap).cuda(), out=want)
    n = {b.GS_TENSOR: 1, b.GS_ROW: D, b.GS_BLOCK128: D * (got.Kp // 128)}[gs]
    assert torch.equal(got.gscale[:n], want.gscale[:n])
    assert np.array_equal(got.sf_linear(), want.sf_linear())
    assert torch.equal(got.codes[: D * got.Kp // 2], want.codes[: D * got.Kp // 2])
