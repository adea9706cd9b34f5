"""The calls behind the captures of single kernels: each kernel of interest once, on tensors beyond the L2 or at a layer's own sizes.

ncu --clock-control none -k regex:"<names>" --metrics <metrics> --csv --log-file calls.csv python profiles/single_calls.py [group ...]
"""
import os
import sys

import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
from paper_2510_27527_b200 import binding as b, synth  # noqa: E402

SR, RTN, ROW, COL = b.ROUND_SR, b.ROUND_RTN, b.AXIS_ROW, b.AXIS_COL


def mk(rows, cols, scale=1.0):
    return (torch.randn(rows, cols, device="cuda") * scale).to(torch.bfloat16)


def quantizers(gs):
    x = mk(8192, 8192)
    q = b.nvfp4_quantize(x, ROW, RTN, 1, 1, gs)
    b.nvfp4_quantize(x, ROW, SR, 1, 3, gs)
    b.nvfp4_quantize(x, COL, SR, 1, 5, gs)
    b.nvfp4_requantize_t(q, SR, 1, 6, gs)


def hadamard():
    dy, x = mk(8192, 3072), mk(8192, 1024)
    keep = b.LayerConfig(outliers=synth.outlier_channels(1024, 102, 1)).index(1024)[1]
    b.nvfp4_quantize(dy, ROW, SR, 1, 3, b.GS_BLOCK128, rht_stream_id=7)
    b.nvfp4_quantize(dy, COL, SR, 1, 5, b.GS_BLOCK128, rht_stream_id=8)
    b.nvfp4_requantize_t(b.nvfp4_quantize(x, ROW, RTN, 1, 1, b.GS_BLOCK128, keep_cols=keep), SR, 1, 6, rht_stream_id=8)


def oscillation():
    w = torch.randn(8192, 8192, device="cuda") * 0.02
    other = w + 4e-5 * torch.randn_like(w)
    state = b.alloc_osci_state(w)
    for t0 in range(4):
        b.nvfp4_osci_update(other if t0 & 1 else w, state, t0)
    b.nvfp4_osci_suppress(w, state, 8.0)


def outliers():
    for D, C, n in ((1024, 3072, 102), (1024, 1024, 102), (2816, 1024, 282)):
        x, w, dy = mk(8192, D), mk(C, D, 0.02), mk(8192, C, 1e-4)
        cfg = b.LayerConfig(outliers=synth.outlier_channels(D, n, 1), concurrent=False)
        _, saved = b.nvfp4_linear_fwd(x, w, cfg)
        b.nvfp4_linear_bwd(dy, saved, cfg)


def fp6():
    x = mk(16384, 4096)
    b.nvfp4_fp6_requantize_t(b.nvfp4_fp6_quantize(x, RTN, 1, 1), SR, 1, 6)
    b.nvfp4_fp6_quantize(x, SR, 1, 3)
    b.nvfp4_expand_operand(b.nvfp4_quantize(x, ROW, RTN, 1, 2))
    for m, n, k in ((4096, 3072, 1024), (8192, 8192, 8192)):
        b.nvfp4_dense_gemm(b.nvfp4_fp6_quantize(mk(m, k)), b.nvfp4_fp6_quantize(mk(n, k)), b.DT_BF16)
    b.nvfp4_dense_gemm(b.nvfp4_fp6_quantize(mk(3072, 4096)), b.nvfp4_fp6_quantize(mk(1024, 4096)), b.DT_F32)


GROUPS = {"tensor": lambda: quantizers(b.GS_TENSOR), "block128": lambda: quantizers(b.GS_BLOCK128), "hadamard": hadamard,
          "oscillation": oscillation, "outliers": outliers, "fp6": fp6}
for name in sys.argv[1:] or GROUPS:
    torch.manual_seed(1)
    GROUPS[name]()
    torch.cuda.synchronize()
print("done")
