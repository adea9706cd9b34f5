"""torch.autograd wrapper around the C-ABI layer calls: `NVFP4Linear` is a drop-in `nn.Linear` (no bias inside the FP4
product; an optional bias is added in BF16) whose forward is `nvfp4_linear_fwd` and whose backward is `nvfp4_linear_bwd`
(paper Sec. 2.3: Y = Q1(X) Q2(W)^T, dX = Q3(dY) Q4(W-hat), dW = Q5(dY^T) Q6(X-hat)). Argument marshalling only: every step
of the path runs in the library's kernels. The stochastic-rounding key of a call is derived from the configuration's base
seed, the module instance and the call number, so that neither two steps of one layer nor two layers of a model built
from the same configuration share their draws.
"""
from __future__ import annotations

import ctypes
import functools

import torch
from torch.autograd import forward_ad

from . import binding as B
from .build import node_tag

try:
    from . import _node
    if getattr(_node, "built_for", None) != node_tag():  # (it may load all the same)
        raise ImportError(f"{_node.__file__} is not for {node_tag()}")
except ImportError as e:
    raise ImportError(f"{e}: build it with `python -m paper_2510_27527_b200.build`") from e


_MASK64 = (1 << 64) - 1


def call_seed(base_seed: int, layer_id: int, call: int) -> int:
    """64-bit Philox key of one forward / backward call: a fixed mixing (splitmix64 finaliser) of the base seed, the module
    instance and the call number. Distinct (layer, call) pairs give distinct, unrelated keys; layers of equal shape would
    otherwise draw identical stochastic-rounding bits element for element."""
    z = (base_seed + 0x9E3779B97F4A7C15 * (layer_id + 1) + 0xD1B54A32D192ED03 * (call + 1)) & _MASK64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _MASK64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _MASK64
    return z ^ (z >> 31)


def _up(n: int) -> int:
    return (n + 255) // 256 * 256


@functools.lru_cache(maxsize=1024)
def _layout(N_tok: int, D: int, C: int, n_out: int, gs_mode: int):
    """Where a call keeps what forward leaves for backward, inside one buffer: the byte offsets of codes, scales and global
    scales of qx and qw and of the two compact outlier matrices (-1: none), the offset and size of forward's workspace, the
    buffer's total, and the size of backward's workspace. Sizes only: no memory is kept."""
    Dk, Kh, at, offs = D - n_out, B.lib.nvfp4_outlier_pad(n_out), 0, []
    for R in (N_tok, C):
        for n in (B.lib.nvfp4_operand_codes_bytes(R, Dk), B.lib.nvfp4_operand_sf_bytes(R, Dk, B.SF_TILED128x4),
                  4 * B.lib.nvfp4_operand_gscale_count(R, Dk, gs_mode)):
            offs.append(at)
            at = _up(at + n)
    for R in (N_tok, C):
        offs.append(at if Kh else -1)
        at = _up(at + R * Kh * 2)
    ws_fwd = B.lib.nvfp4_linear_workspace_bytes(B.OP_FWD, N_tok, D, C, n_out, gs_mode)
    return tuple(offs), at, ws_fwd, at + ws_fwd, B.lib.nvfp4_linear_workspace_bytes(B.OP_BWD, N_tok, D, C, n_out, gs_mode)


class _Call:
    """One forward call and, later, its backward, through the binding: what `_node.linear` does, where it cannot go (`_plain`). Everything
    that is saved lies in one buffer."""

    __slots__ = ("buf", "saved", "ccfg", "keeps", "concurrent", "shape", "ws_bwd")

    def forward(self, x: torch.Tensor, weight: torch.Tensor, cfg: B.LayerConfig, seed: int) -> torch.Tensor:
        (N_tok, D), C, dev = x.shape, weight.shape[0], x.device
        if type(N_tok) is not int:  # (under jit.trace sizes are tensors)
            N_tok, D, C = int(N_tok), int(D), int(C)
        index = cfg.index(D, dev)
        n_out, gs = cfg.n_out, cfg.gs_mode
        offs, ws_at, ws_fwd, total, self.ws_bwd = _layout(N_tok, D, C, n_out, gs)
        buf = torch.empty(total, dtype=torch.uint8, device=dev)
        y = B._matrix(N_tok, C, B.DT_BF16, dev)
        p, stream = buf.data_ptr(), B._stream_ptr()
        at = [p + o if o >= 0 else 0 for o in offs]
        saved = B.CSaved(B.COperand(at[0], at[1], at[2], N_tok, D - n_out, gs, B.SF_TILED128x4),
                         B.COperand(at[3], at[4], at[5], C, D - n_out, gs, B.SF_TILED128x4), X_out=at[6], W_out=at[7])
        # the configuration as it is now: what the caller changes later belongs to later calls
        ccfg = cfg.c(index, seed, (B.DT_BF16, B.DT_BF16, B.DT_BF16), B.thread_side(dev, stream) if cfg.concurrent else None)
        B._check(B.lib.nvfp4_linear_fwd(x.data_ptr(), x.stride(0), weight.data_ptr(), weight.stride(0), N_tok, D, C, ctypes.byref(ccfg),
                                        y.data_ptr(), y.stride(0), ctypes.byref(saved), p + ws_at, ws_fwd, stream), "nvfp4_linear_fwd")
        self.buf, self.saved, self.ccfg, self.shape = buf, saved, ccfg, (N_tok, D, C)
        self.keeps, self.concurrent = (index, cfg.dev_status), cfg.concurrent
        return y

    def backward(self, dy: torch.Tensor):
        (N_tok, D, C), dev = self.shape, dy.device
        dx, dw = B._matrix(N_tok, D, B.DT_BF16, dev), B._matrix(C, D, B.DT_BF16, dev)
        ws, stream = torch.empty(self.ws_bwd, dtype=torch.uint8, device=dev), B._stream_ptr()
        ccfg = B.CLayerCfg.from_buffer_copy(self.ccfg)
        if self.keeps[0] is not None:
            self.keeps[0].here()
        if self.concurrent:  # autograd runs backward on a thread of its own, which has its own second stream and events
            B.set_side(ccfg, B.thread_side(dev, stream))
        B._check(B.lib.nvfp4_linear_bwd(dy.data_ptr(), dy.stride(0), ctypes.byref(self.saved), ctypes.byref(ccfg), dx.data_ptr(), dx.stride(0),
                                        dw.data_ptr(), dw.stride(0), ws.data_ptr(), self.ws_bwd, stream), "nvfp4_linear_bwd")
        return dx, dw


def _plain(x: torch.Tensor, weight: torch.Tensor) -> bool:
    """Whether a call can go to the native node. Not while a trace is recorded or compiled (it would not see what the library writes), under
    forward-mode differentiation or a function transform (which the autograd function refuses), or with tensor subclasses."""
    return (not torch.compiler.is_compiling() and type(x) is torch.Tensor and type(weight) is torch.nn.Parameter and forward_ad._current_level < 0
            and not torch._C._is_tracing() and not torch._C._are_functorch_transforms_active())


def _needs_function(x: torch.Tensor, weight: torch.Tensor) -> bool:
    """Whether a call that the native node does not serve has to go through the autograd function: a gradient can be asked for, an input may
    carry a forward-mode tangent or be a transform's (which the function refuses), or a trace is being recorded (which sees the function, but
    not what the library writes). Else it goes to the library at once (48 instead of 55 us on 77 tokens)."""
    return ((torch.is_grad_enabled() and (x.requires_grad or weight.requires_grad)) or forward_ad._current_level >= 0 or torch.jit.is_tracing()
            or torch._C._are_functorch_transforms_active())


class _NVFP4LinearFn(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x2d: torch.Tensor, weight: torch.Tensor, cfg: B.LayerConfig, seed: int):
        ctx.call = _Call()
        return ctx.call.forward(x2d, weight, cfg, seed)

    @staticmethod
    def backward(ctx, dy: torch.Tensor):
        dy = dy.contiguous()
        if dy.dtype != torch.bfloat16:
            dy = dy.to(torch.bfloat16)
        dx, dw = ctx.call.backward(dy)
        return dx, dw, None, None


class NVFP4Linear(torch.nn.Module):
    """y = x W^T (+ bias) with the NVFP4 forward and backward products. Inputs and weights are BF16 on a CUDA device."""

    _instances = 0  # every module takes the next id: its own stream of stochastic-rounding keys

    def __init__(self, in_features: int, out_features: int, bias: bool = False, cfg: B.LayerConfig | None = None, device="cuda"):
        super().__init__()
        self.in_features, self.out_features = in_features, out_features
        self.weight = torch.nn.Parameter(torch.empty(out_features, in_features, dtype=torch.bfloat16, device=device))
        torch.nn.init.normal_(self.weight, std=0.02)
        self.bias = torch.nn.Parameter(torch.zeros(out_features, dtype=torch.bfloat16, device=device)) if bias else None
        self.cfg = cfg if cfg is not None else B.LayerConfig()
        self._calls = 0
        self.layer_id = NVFP4Linear._instances
        NVFP4Linear._instances += 1

    def forward(self, x: torch.Tensor) -> torch.Tensor:
        shape, weight = x.shape, self.weight
        if len(shape) == 0 or shape[-1] != self.in_features:  # the library takes a narrower input with the weights' leading dimension
            raise RuntimeError(f"NVFP4Linear: input of shape {tuple(shape)} for {self.in_features} input features")
        x2d = x if len(shape) == 2 else x.reshape(-1, self.in_features)
        if x2d.dtype != torch.bfloat16:
            x2d = x2d.to(torch.bfloat16)
        x2d = x2d.contiguous()
        # this layer's key of this call
        seed = call_seed(self.cfg.seed, self.layer_id, self._calls)
        self._calls += 1
        if _plain(x2d, weight):
            cfg = self.cfg
            index = None if cfg.outliers is None else cfg.index(self.in_features, x2d.device)
            y = _node.linear(x2d, weight, cfg, index, seed, torch.is_grad_enabled() and (x2d.requires_grad or weight.requires_grad))
        elif _needs_function(x2d, weight):
            y = _NVFP4LinearFn.apply(x2d, weight, self.cfg, seed)
        else:
            y = _Call().forward(x2d, weight, self.cfg, seed)
        if self.bias is not None:
            y = y + self.bias
        return y if len(shape) == 2 else y.reshape(*shape[:-1], self.out_features)
