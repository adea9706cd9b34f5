"""The FP6 row quantizer's two forms of the tensor maximum (64 words, one cleared word) and one or four blocks per thread: every value and
scale is the same, whatever the workspace holds and whichever form the size takes."""

import numpy as np
import pytest
import torch

from paper_2510_27527_b200 import binding as b

pytestmark = pytest.mark.gpu

# Blocks of the padded output around the lines: 148 * 4 * 256 = 151552 (one or four per thread, to nearest), 148 * 8 * 256 = 303104 and
# 2^20 (words or one word, to nearest and stochastic); rows that end inside a block, a row of one block, and a tensor smaller than one CTA.
SHAPES = [(1, 8), (3, 24), (77, 1000), (2368, 1024), (2369, 1024), (4736, 1024), (4737, 1016), (8192, 2048), (8193, 2048), (151553, 16)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("rounding", [0, 1])
def test_every_form_gives_the_same_operand(shape, rounding):
    rows, cols = shape
    gen = torch.Generator(device="cuda").manual_seed(rows * 31 + cols)
    full = torch.randn(rows, cols + 8, generator=gen, device="cuda", dtype=torch.bfloat16)
    full[rows // 2, 0] = -37.0  # the maximum, once, in the first column
    src = full[:, :cols]
    got = []
    for nbytes in (16, 128, 256, 4096):
        ws = torch.full((nbytes,), 0x7F, dtype=torch.uint8, device="cuda")
        out = b.alloc_dense(rows, cols, poison=True)
        b.nvfp4_fp6_quantize(src, rounding, 4242, 3, out=out, workspace=ws)
        got.append(out)
    assert float(got[0].gscale[0]) == float(np.float32(37.0) / np.float32(3360.0))
    for g in got[1:]:
        assert torch.equal(g.vals.view(torch.int16), got[0].vals.view(torch.int16)) and torch.equal(g.gscale, got[0].gscale)
    # a value is x to half a step of E2M3 (2^-4 of it) and of the block scale (2^-4 of it), one step under stochastic rounding: the sum
    # of both, below 3/16 of x plus 1/4 of a step (7.5 S is the block's largest, S at most its maximum / 7)
    x = src.float()
    y = got[0].vals[:, :cols].float() * got[0].gscale
    pad = torch.nn.functional.pad(x.abs(), (0, -cols % 16)).reshape(rows, -1, 16).amax(2).repeat_interleave(16, 1)[:, :cols]
    assert bool(((y - x).abs() <= x.abs() * 0.1875 + pad * (0.25 / 7)).all())


@pytest.mark.parametrize("rounding", [0, 1])
def test_the_librarys_own_workspace_size_saves_the_clearing_launch(rounding):
    x = torch.randn(64, 256, device="cuda").to(torch.bfloat16)
    out = b.alloc_dense(64, 256)

    def launches(nbytes):
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        before = b.lib.nvfp4_launch_count()
        b.nvfp4_fp6_quantize(x, rounding, 1, 1, out=out, workspace=ws)
        return b.lib.nvfp4_launch_count() - before

    assert launches(b.lib.nvfp4_fp6_workspace_bytes()) == 2 and launches(16) == 3
    with pytest.raises(b.Nvfp4Error, match="workspace"):
        launches(15)
