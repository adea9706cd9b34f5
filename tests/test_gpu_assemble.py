"""The pass that puts a weight gradient together from the compact product of the kept channels and the token splits of the outlier
channels: at widths that take its rows through shared memory four at a time, two at a time and not at all, and at ragged rows."""
import numpy as np
import pytest
import torch

from paper_2510_27527_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,D,C", [(64, 264, 5), (300, 1000, 133), (2048, 512, 8), (64, 8200, 6), (64, 20000, 5)])
@pytest.mark.parametrize("n_out", [1, 66])
@pytest.mark.parametrize("f32", [True, False])
def test_weight_gradient_of_kept_and_outlier_channels(T, D, C, n_out, f32):
    from paper_2510_27527_b200 import binding as b

    g = torch.Generator(device="cuda").manual_seed(D + n_out)
    mk = lambda r, c: torch.randn(r, c, device="cuda", generator=g).to(torch.bfloat16)  # noqa: E731
    x, w, dy = mk(T, D), mk(C, D), mk(T, (C + 7) // 8 * 8)[:, :C]
    outl = synth.outlier_channels(D, n_out, 9)
    keep = torch.from_numpy(np.setdiff1d(np.arange(D), outl)).cuda()
    cfg = b.LayerConfig(gs_mode=b.GS_TENSOR, seed=5, outliers=outl, dw_dtype=b.DT_F32 if f32 else b.DT_BF16)
    _, saved = b.nvfp4_linear_fwd(x, w, cfg)
    ws = b.linear_workspace(b.OP_BWD, T, D, C, cfg)
    ld = (D + 7) // 8 * 8 + 8
    buf = torch.full((C, ld), 77.0, dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
    dw = buf[:, :D]
    b.nvfp4_linear_bwd(dy, saved, cfg, dW=dw, workspace=ws)
    q5, q6 = (b.nvfp4_linear_bwd_operand(b.OP_BWD, i, T, D, C, cfg, ws) for i in (5, 6))
    kept = b.nvfp4_gemm(q5, q6, b.DT_F32)  # the same product: the same bits
    assert torch.equal(dw[:, keep], kept if f32 else kept.to(torch.bfloat16))
    idx = torch.from_numpy(np.asarray(outl)).cuda()
    want = dy.double().T @ x[:, idx].double()
    absdot = dy.double().abs().T @ x[:, idx].double().abs()
    # exact products summed in FP32: at most T roundings of 2^-24 of the sum of magnitudes; then one of BF16
    tol = T * 2.0 ** -24 * absdot + (0.0 if f32 else 2.0 ** -8 * want.abs())
    assert bool(((dw[:, idx].double() - want).abs() <= tol).all())
    assert bool((buf[:, D:] == 77.0).all())


@pytest.mark.parametrize("D,n_out", [(264, 5), (1000, 300), (8200, 66), (20000, 1)])
def test_an_outlier_takes_its_sums_whatever_the_channel_map_holds_for_it(D, n_out):
    from paper_2510_27527_b200 import binding as b

    g = torch.Generator(device="cuda").manual_seed(D)
    mk = lambda r, c: torch.randn(r, c, device="cuda", generator=g).to(torch.bfloat16)  # noqa: E731
    x, w, dy = mk(128, D), mk(16, D), mk(128, 16)
    cfg = b.LayerConfig(gs_mode=b.GS_TENSOR, seed=5, outliers=synth.outlier_channels(D, n_out, 9))
    _, saved = b.nvfp4_linear_fwd(x, w, cfg)
    want = b.nvfp4_linear_bwd_dw(dy, saved, cfg)
    outl, _, cmap = saved.index
    for value in (0, D - n_out - 1):  # positions of kept channels
        cmap[outl.long()] = value
        for _ in range(5):
            assert torch.equal(b.nvfp4_linear_bwd_dw(dy, saved, cfg), want)
