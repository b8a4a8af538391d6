"""Straight-through FP4 linear layer on top of the C-ABI calls (glue only; every step runs in the library's kernels).

Section 3.1 of the paper: the forward product uses 2D-block-quantized weights and activations (round to nearest),
the backward pass quantizes the incoming gradient once (stochastic rounding) and uses it, with the quantized
operands saved by the forward pass, in both backward products; the quantizers are treated as identity when
differentiating (straight-through estimator).  Because the blocks are 32x32, the transposed payloads the backward
products need are written by the same quantization call: nothing is re-quantized between forward and backward.
"""
from __future__ import annotations

import torch
from torch.autograd import forward_ad

from . import binding


class _FP4LinearFn(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x, weight, seed, tensor_id, ws):
        # x [T, K], weight [N, K]; both are quantized once, with both payload layouts
        qx = binding.fp4q_quantize2d(x.to(torch.bfloat16).contiguous(), mode=binding.ROUND_NEAREST)
        qw = binding.fp4q_quantize2d(weight.to(torch.bfloat16).contiguous(), mode=binding.ROUND_NEAREST)
        y = binding.fp4q_gemm_fwd(qx, qw, dt=binding.OUT_BF16, ws=ws)
        ctx.qx, ctx.qw, ctx.ws = qx, qw, ws
        ctx.seed, ctx.tensor_id = int(seed), int(tensor_id)
        ctx.x_dtype, ctx.w_dtype = x.dtype, weight.dtype
        return y if y.is_contiguous() else y.contiguous()

    @staticmethod
    def backward(ctx, dy):
        qdy = binding.fp4q_quantize2d(dy.to(torch.bfloat16).contiguous(), mode=binding.ROUND_STOCHASTIC,
                                      seed=ctx.seed, tensor_id=ctx.tensor_id)
        dx = dw = None
        if ctx.needs_input_grad[0]:
            dx = binding.fp4q_gemm_dgrad(qdy, ctx.qw, dt=binding.OUT_BF16, ws=ctx.ws).to(ctx.x_dtype)
        if ctx.needs_input_grad[1]:
            dw = binding.fp4q_gemm_wgrad(qdy, ctx.qx, dt=binding.OUT_F32, ws=ctx.ws).to(ctx.w_dtype)
        ctx.qx = ctx.qw = None
        return dx, dw, None, None, None


_TENSORS = (torch.Tensor, torch.nn.Parameter)


def _find_observers():
    """A function that says whether anything looks into Python autograd functions just now: tracers, transforms, modes, forward-mode
    levels.  None where this torch lacks one of the names, which are not public."""
    try:
        compiling, tracing = torch.compiler.is_compiling, torch._C._get_tracing_state
        transforms, dispatch, function = torch._C._functorch.peek_interpreter_stack, torch._C._len_torch_dispatch_stack, torch._C._len_torch_function_stack
        forward_ad._current_level   # a variable: read at every call
    except AttributeError:
        return None

    def observed() -> bool:
        return (compiling() or transforms() is not None or dispatch() != 0 or function() != 0 or tracing() is not None
                or forward_ad._current_level >= 0)
    return observed


_observed = _find_observers()


def _plain(x, weight) -> bool:
    """Ordinary tensors on one GPU and nothing that looks into a Python autograd function: the native node does the same in half
    the host's time.  Everything else, what is refused included, goes through _FP4LinearFn."""
    return (_observed is not None and type(x) in _TENSORS and type(weight) in _TENSORS and x.is_cuda and weight.dim() == 2
            and x.device == weight.device and not _observed())


def _linear(x, weight, seed, tensor_id, ws):
    if _plain(x, weight):
        return binding._host().linear(x, weight, int(seed), int(tensor_id), ws)
    return _FP4LinearFn.apply(x, weight, seed, tensor_id, ws)


def fp4_linear(x: torch.Tensor, weight: torch.Tensor, seed: int = 0, tensor_id: int = 0, ws=None) -> torch.Tensor:
    """y = x^ weight^^T with FP4 forward and backward products.  x [..., K] and weight [N, K] live on the GPU;
    `seed` / `tensor_id` key the stochastic rounding of the incoming gradient (change one of them every step)."""
    if ws is None:
        ws = binding.alloc_workspace(x.device)
    if x.dim() == 2 and x.shape[1] != 0:   # nothing to fold: two autograd nodes less (reshape refuses rows of nothing)
        return _linear(x, weight, seed, tensor_id, ws)
    lead = x.shape[:-1]
    y = _linear(x.reshape(-1, x.shape[-1]), weight, seed, tensor_id, ws)
    return y.reshape(*lead, weight.shape[0])


class FP4Linear(torch.nn.Module):
    """Bias-free linear layer with an FP32 master weight and FP4 products.  Each backward pass draws fresh
    stochastic-rounding bits: the module counts its forward calls and uses the count as the Philox tensor id's
    high part, `layer_id` as the low 8 bits."""

    def __init__(self, in_features: int, out_features: int, layer_id: int = 0, seed: int = 0, device="cuda"):
        super().__init__()
        self.weight = torch.nn.Parameter(torch.empty(out_features, in_features, device=device, dtype=torch.float32))
        torch.nn.init.normal_(self.weight, std=0.02)
        self.layer_id, self.seed, self.calls = int(layer_id) & 0xFF, int(seed), 0
        self._ws = None

    def forward(self, x: torch.Tensor) -> torch.Tensor:
        if self._ws is None or self._ws.device != x.device:
            self._ws = binding.alloc_workspace(x.device)
        self.calls += 1
        tid = ((self.calls & 0xFFFFFF) << 8) | self.layer_id
        return fp4_linear(x, self.weight, seed=self.seed, tensor_id=tid, ws=self._ws)
