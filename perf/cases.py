"""What a training or evaluation program has the NVFP4 linear layer do, as cases whose speed is measured.

Shapes are those of the repository's own configurations: the 24-layer model of hidden size 1024 and FFN size 2816, its
attention and MLP projections at 8192 and 16384 tokens, the single 512-wide layer, the quantize-and-multiply sweep up to
16384 x 8192 x 8192, and ragged sizes as in the tests. Inputs follow the same recipe as the synthetic tensors of the package
(activations ~N(0, 1) with a few channels scaled up, silu(g) * u for down projections, weights ~N(0, 0.02), Student-t
gradients with three degrees of freedom), drawn on the device from the seed.

Kinds of case:
  module     NVFP4Linear, a drop-in nn.Linear: forward and, with "train", backward through autograd. Nothing is kept between
             steps but the module (buffers come from torch's allocator on every call).
  linears    several linears of a block through nvfp4_linear_fwd / nvfp4_linear_bwd with outputs, saved operands and workspaces
             kept from step to step, as a training loop that owns its memory does.
  matmul     nvfp4_quantize of an activation matrix and nvfp4_gemm with weights that were quantized once.
  osci       one step of the oscillation statistics on the FP32 master weights of a block, and the reset that follows.
  calibrate  one step of the outlier-channel calibration and the choice of channels.
  fp6        the simulated FP6 x FP4 layer, forward and backward.
"""
import math

import numpy as np
import torch

from paper_2510_27527_b200 import binding as B
from paper_2510_27527_b200.module import NVFP4Linear

GS = {"tensor": B.GS_TENSOR, "row": B.GS_ROW, "block128": B.GS_BLOCK128}

# "in x out" of the linears of one block of the 370M model; "s" marks an input that is silu(g) * u
ATTENTION = "1024x3072 1024x1024"
MLP = "1024x2816 1024x2816 2816x1024s"
BLOCK = ATTENTION + " " + MLP


def listed():
    return [
        # the smallest training step: one 512-wide layer on a batch of 256 tokens, where launches and host work are what counts
        dict(name="layer_256", kind="module", train=True, tokens=256, shapes="512x512", gs="tensor", rht=False, outliers=0.0),
        # evaluation of a short prompt of odd length, forward only
        dict(name="prompt_77", kind="module", train=False, tokens=77, shapes="1024x3072", gs="tensor", rht=False, outliers=0.0),
        # an ordinary step of one projection: 4 sequences of 2048 tokens, default options
        dict(name="qkv_8192", kind="module", train=True, tokens=8192, shapes="1024x3072", gs="tensor", rht=False, outliers=0.0),
        # all linears of a block of the 370M model, 8 sequences of 2048 tokens: what a step of pre-training consists of
        dict(name="block_16384", kind="linears", train=True, tokens=16384, shapes=BLOCK, gs="tensor", rht=False, outliers=0.0),
        # the paper's base recipe (1x128 outer blocks, Hadamard transformation in backward) on a block at the smaller batch
        dict(name="block_paper_8192", kind="linears", train=True, tokens=8192, shapes=BLOCK, gs="block128", rht=True, outliers=0.0),
        # the paper's full recipe (with 10 % of the channels in BF16) on the MLP
        dict(name="mlp_full_recipe_8192", kind="linears", train=True, tokens=8192, shapes=MLP, gs="block128", rht=True, outliers=0.1),
        # outlier channels under per-tensor scales, on a batch whose token count is odd
        dict(name="gate_outliers_4095", kind="module", train=True, tokens=4095, shapes="1024x2816", gs="tensor", rht=False, outliers=0.1),
        # per-row scales on ragged sizes
        dict(name="ragged_rows_1999", kind="module", train=True, tokens=1999, shapes="1000x1416", gs="row", rht=False, outliers=0.0),
        # the largest product of the sweep, with the quantization of its activations
        dict(name="matmul_16384_8192_8192", kind="matmul", tokens=16384, shapes="8192x8192", gs="tensor"),
        # oscillation suppression on the weights of a block, one statistics step and one reset
        dict(name="osci_block", kind="osci", shapes=BLOCK, gs="tensor", sparse=False),
        # outlier-channel calibration on the input of the MLP
        dict(name="calibrate_16384", kind="calibrate", tokens=16384, shapes="1024x2816", outliers=0.1),
        # the precision-switching study's layer
        dict(name="fp6_qkv_4096", kind="fp6", train=True, tokens=4096, shapes="1024x3072"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _width(rng, lo=256, hi=4096):
    return int(_log(rng, lo, hi)) // 8 * 8


def draw(rng):
    """One more case of these ranges: tokens 64 .. 16384 of any parity, widths 256 .. 4096 (multiples of 8), every option."""
    kind = rng.choice(["module", "module", "module", "linears", "linears", "linears", "matmul", "osci", "calibrate", "fp6"])
    tokens = int(_log(rng, 64, 16384.5))
    if rng.random() < 0.25:  # whole sequences
        tokens = max(64, tokens // 256 * 256)
    D, C = _width(rng), _width(rng)
    gs = rng.choice(["tensor", "tensor", "block128", "row"])
    if kind in ("module", "linears"):
        train = kind == "linears" or rng.random() < 0.75
        shapes, most = "%dx%d" % (D, C), 2 * D * C
        if kind == "linears":  # an MLP of these sizes (D the narrower), or two projections
            d, c = min(D, C, 2048), max(D, C)
            shapes, most = rng.choice([("%dx%d %dx%ds" % (d, c, c, d), 2 * d * c), ("%dx%d %dx%d" % (d, c, d, d), d * c + d * d)])
        # no more than a step of the listed blocks
        tokens = min(tokens, int((1.2e12 if gs == "tensor" else 0.5e12) / 6 / most))
        return dict(kind=kind, train=train, tokens=tokens, shapes=shapes, gs=gs, rht=rng.random() < 0.4,
                    outliers=rng.choice([0.0, 0.0, 0.0, 0.01, 0.05, 0.1]))
    if kind == "matmul":
        D, C = _width(rng, 256, 8192), _width(rng, 256, 8192)
        tokens = min(tokens, int((2.2e12 if gs == "tensor" else 0.5e12) / 2 / (D * C)))
        return dict(kind=kind, tokens=tokens, shapes="%dx%d" % (D, C), gs=gs)
    if kind == "osci":
        return dict(kind=kind, shapes="%dx%d" % (D, C), gs=gs, sparse=rng.random() < 0.5)
    if kind == "calibrate":
        return dict(kind=kind, tokens=tokens, shapes="%dx%d" % (D, C), outliers=rng.choice([0.01, 0.05, 0.1]))
    return dict(kind=kind, train=True, tokens=min(tokens, 4096), shapes="%dx%d" % (min(D, 2048), min(C, 2048)))


def _shapes(case):
    """[(inputs D, outputs C, silu(g) * u input?)] of the case's linears."""
    out = []
    for s in case["shapes"].split():
        d, c = s.rstrip("s").split("x")
        out.append((int(d), int(c), s.endswith("s")))
    return out


def _activations(g, tokens, D, swiglu, n_hot=10, factor=30.0):
    x = torch.randn(tokens, D, generator=g, device="cuda")
    if swiglu:
        x = torch.nn.functional.silu(x) * torch.randn(tokens, D, generator=g, device="cuda")
    hot = torch.randperm(D, generator=g, device="cuda")[:n_hot]
    x[:, hot] *= factor
    return x.to(torch.bfloat16)


def _weights(g, C, D):
    return (torch.randn(C, D, generator=g, device="cuda") * 0.02).to(torch.bfloat16)


def _gradients(g, tokens, C, scale=1e-4):
    t = torch.randn(tokens, C, generator=g, device="cuda")
    s = torch.zeros(tokens, C, device="cuda")
    for _ in range(3):
        s += torch.randn(tokens, C, generator=g, device="cuda").square_()
    return (t * (s / 3.0).rsqrt_() * scale).to(torch.bfloat16)


def _config(case, D, seed):
    n_out = int(round(case["outliers"] * D))
    outl = np.sort(np.random.default_rng(seed).choice(D, size=n_out, replace=False)) if n_out else None
    return B.LayerConfig(gs_mode=GS[case["gs"]], seed=seed, rht=case["rht"], outliers=outl)


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "module":
        (D, C, _), = _shapes(case)
        layer = NVFP4Linear(D, C, cfg=_config(case, D, seed))
        layer.layer_id = 0  # its place in the model, which keys the random draws: not how many modules the process has made
        with torch.no_grad():
            layer.weight.copy_(_weights(g, C, D))
        x = _activations(g, case["tokens"], D, False)
        if not case["train"]:
            return dict(kind=kind, train=False, layer=layer, x=x)
        return dict(kind=kind, train=True, layer=layer, x=x.requires_grad_(), dy=_gradients(g, case["tokens"], C))
    if kind == "linears":
        return dict(kind=kind, linears=[_linear(case, g, case["tokens"], D, C, s, seed + i) for i, (D, C, s) in enumerate(_shapes(case))])
    if kind == "matmul":
        (D, C, _), = _shapes(case)
        gs = GS[case["gs"]]
        return dict(kind=kind, gs=gs, x=_activations(g, case["tokens"], D, False, max(1, D // 200), 100.0),
                    qx=B.alloc_operand(case["tokens"], D, gs), qw=B.nvfp4_quantize(_weights(g, C, D), gs_mode=gs),
                    y=torch.empty(case["tokens"], C, dtype=torch.bfloat16, device="cuda"), ws=torch.empty(1 << 20, dtype=torch.uint8, device="cuda"))
    if kind == "osci":
        return dict(kind=kind, gs=GS[case["gs"]], sparse=case["sparse"],
                    weights=[_master_weights(g, C, D, GS[case["gs"]], case["sparse"]) for D, C, _ in _shapes(case)])
    if kind == "calibrate":
        (D, _, _), = _shapes(case)
        x = _activations(g, case["tokens"], D, False)
        # the window of a few earlier steps
        acc = torch.rand(D, generator=g, device="cuda") + 3.0 * math.sqrt(case["tokens"])
        return dict(kind=kind, x=x, acc=acc, n_out=max(1, int(round(case["outliers"] * D))),
                    ws=torch.empty(B.lib.nvfp4_outlier_accumulate_workspace_bytes(case["tokens"], D), dtype=torch.uint8, device="cuda"))
    (D, C, _), = _shapes(case)
    return dict(kind=kind, seed=seed, x=_activations(g, case["tokens"], D, False), w=_weights(g, C, D), dy=_gradients(g, case["tokens"], C))


def _linear(case, g, tokens, D, C, swiglu, seed):
    cfg = _config(case, D, seed)
    cfg.prepare(D)
    x, w, dy = _activations(g, tokens, D, swiglu), _weights(g, C, D), _gradients(g, tokens, C)
    mk = lambda r, c, t: torch.empty(r, c, dtype=t, device="cuda")  # noqa: E731
    return dict(cfg=cfg, x=x, w=w, dy=dy, saved=B.alloc_saved(x, w, cfg), y=mk(tokens, C, torch.bfloat16), dx=mk(tokens, D, torch.bfloat16),
                dw=mk(C, D, torch.float32), ws_fwd=B.linear_workspace(B.OP_FWD, tokens, D, C, cfg),
                ws_bwd=B.linear_workspace(B.OP_BWD, tokens, D, C, cfg))


def _master_weights(g, C, D, gs, sparse):
    """FP32 master weights at two optimizer steps; a few per cent of the elements oscillate by 1.5 % of their value."""
    w0 = torch.randn(C, D, generator=g, device="cuda") * 0.02
    osc = torch.rand(C, D, generator=g, device="cuda") < 0.02
    w1 = w0 + torch.randn(C, D, generator=g, device="cuda") * 4e-5 + osc * 0.015 * w0.abs()
    if sparse:
        state = B.alloc_osci_sparse_state(max(1, C * D // 20))
        ws = torch.empty(max(B.lib.nvfp4_osci_sparse_workspace_bytes(C, D, gs, state.idx.numel(), k) for k in (0, 1, 2)), dtype=torch.uint8, device="cuda")
        B.nvfp4_osci_sparse_update(w0, state, 0, gs, workspace=ws)
    else:
        state = B.alloc_osci_state(w0)
        ws = torch.empty(B.lib.nvfp4_osci_workspace_bytes(C, gs), dtype=torch.uint8, device="cuda")
        B.nvfp4_osci_update(w0, state, 0, gs, workspace=ws)
    return dict(w=w1, state=state, ws=ws, n_reset=torch.zeros(1, dtype=torch.int64, device="cuda"))


def run(s):
    kind = s["kind"]
    if kind == "module":
        if not s["train"]:
            with torch.no_grad():
                return s["layer"](s["x"])
        y = s["layer"](s["x"])
        dx, dw = torch.autograd.grad(y, (s["x"], s["layer"].weight), s["dy"])
        return [y, dx, dw]
    if kind == "linears":
        for l in s["linears"]:
            B.nvfp4_linear_fwd(l["x"], l["w"], l["cfg"], Y=l["y"], saved=l["saved"], workspace=l["ws_fwd"])
        for l in reversed(s["linears"]):
            B.nvfp4_linear_bwd(l["dy"], l["saved"], l["cfg"], dX=l["dx"], dW=l["dw"], workspace=l["ws_bwd"])
        return [(l["y"], l["dx"], l["dw"]) for l in s["linears"]]
    if kind == "matmul":
        B.nvfp4_quantize(s["x"], gs_mode=s["gs"], out=s["qx"], workspace=s["ws"])
        B.nvfp4_gemm(s["qx"], s["qw"], B.DT_BF16, out=s["y"], workspace=s["ws"])
        return [s["y"], s["qx"].codes, s["qx"].sf, s["qx"].gscale]
    if kind == "osci":
        update, suppress = (B.nvfp4_osci_sparse_update, B.nvfp4_osci_sparse_suppress) if s["sparse"] else (B.nvfp4_osci_update, B.nvfp4_osci_suppress)
        for m in s["weights"]:
            update(m["w"], m["state"], 1, s["gs"], workspace=m["ws"])
            suppress(m["w"], m["state"], 6.0, s["gs"], n_reset=m["n_reset"], workspace=m["ws"])
        if s["sparse"]:
            return [(m["w"], m["state"].idx, m["state"].WM_prev, m["state"].WQ_prev, m["state"].D_M, m["state"].D_Q, m["n_reset"]) for m in s["weights"]]
        return [(m["w"], m["state"].W_prev, m["state"].D_M, m["state"].D_Q, m["n_reset"]) for m in s["weights"]]
    if kind == "calibrate":
        B.nvfp4_outlier_accumulate(s["x"], s["acc"], workspace=s["ws"])
        return [s["acc"], *B.nvfp4_outlier_select(s["acc"], s["n_out"])]
    y, saved = B.fp6_linear_fwd(s["x"], s["w"])
    dx, dw, _ = B.fp6_linear_bwd(s["dy"], saved, s["seed"])
    return [y, dx, dw]


def work(case):
    """Bytes read and written once, and the products' operations, of one pass."""
    kind, b, f = case["kind"], 0, 0
    T = case.get("tokens", 0)
    for D, C, _ in _shapes(case):
        if kind in ("module", "linears", "fp6"):
            b += 2 * (T * D + C * D + T * C)
            f += 2 * T * D * C
            if case["train"]:  # dY in, dX out (BF16), dW out (BF16 from the module, else FP32)
                b += 2 * (T * C + T * D) + (2 if kind == "module" else 4) * C * D
                f += 4 * T * D * C
        elif kind == "matmul":  # X in, its operand out, W's operand in, Y out
            b += 2 * T * D + 0.5625 * (T * D + C * D) + 2 * T * C
            f += 2 * T * D * C
        elif kind == "osci":
            if case["sparse"]:  # W once, its tracked twentieth in and out with 20 bytes of state
                b += 4 * C * D + C * D // 20 * 40
            else:  # W and three FP32 state arrays in, three of them and W out
                b += 32 * C * D
        else:
            b += 2 * T * D + 8 * D + 8 * D
    return {"bytes": b, "flops": f}


def tolerance(case):
    if case["kind"] == "osci":
        return "exact"
    if case["kind"] == "calibrate":  # 32-bit sums of squares in another order; channels of equal norm may change places
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
    # the quantized operands are the same bytes; their products' 32-bit sums may run in another order, after which a BF16
    # result can round to its neighbour (2^-7 of its value at most). Against products of the same operands in 64 bits, results
    # in BF16 were 4e-5 off at most (largest single difference 8e-3), those in FP32 2e-7.
    return {"rel": 2e-4, "max": 0.03, "differ": 0.0}
