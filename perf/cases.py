"""The work that users of this library have it do, as timed cases.

A case is one pass of a training layer (or of its quantizers alone) through the public entry points: the
straight-through layer of paper_2607_24953_b200.autograd and the calls of paper_2607_24953_b200.binding.  Sizes
are those of the workload configurations (tiny, 1B-class, 7B-class, query/key projections, expert layer), of the
block-size study and of the tests' ragged shapes; `draw` spreads the same kinds of pass over the ranges between
them.  Inputs have the configurations' value distributions (workloads.py), drawn on the GPU from the seed.
"""
import math
import random

import numpy as np
import torch

from paper_2607_24953_b200 import autograd, binding, workloads

DEVICE = "cuda:0"


def listed():
    return [
        # The smallest layer anyone runs: the tiny linear layer's forward and backward through autograd.  Launches and
        # host time are all there is.
        {"name": "linear tiny", "kind": "linear", "T": 128, "N": 256, "K": 256},
        # A hidden projection of the 1B-class model, FP32 master weight, forward and backward through autograd.
        {"name": "linear 1B", "kind": "linear", "T": 8192, "N": 2048, "K": 2048},
        # Nothing aligned: a packed batch of odd length and odd layer widths (pruned or vocabulary-sized layers), so every
        # tile has an edge and no row of the inputs starts on a vector boundary.
        {"name": "linear ragged", "kind": "linear", "T": 1999, "N": 1003, "K": 2731},
        # The benchmark's layer: gate projection of the 7B-class model, operands quantized with stochastic rounding by one
        # call, then the three products.
        {"name": "layer 7B", "kind": "layer", "T": 16384, "N": 11008, "K": 4096},
        # One microbatch of gradient accumulation: the weight was quantized when the step began, the weight gradient is added
        # to the FP32 sum of the microbatches before it.
        {"name": "microbatch", "kind": "microbatch", "T": 2048, "N": 4096, "K": 4096},
        # Standalone quantize + dual-layout pack of the three operands of the 7B-class down projection, gradient mode.
        {"name": "quantize 7B", "kind": "quantize", "T": 16384, "N": 4096, "K": 11008, "stochastic": True},
        # The same on odd sizes in a row pitch that is no multiple of anything.
        {"name": "quantize ragged", "kind": "quantize", "T": 4099, "N": 1003, "K": 2731, "stochastic": True},
        # Query and key projections in MXFP8 at 7B-class size, and the backward pass of one of them.
        {"name": "qk mxfp8", "kind": "mxfp8", "T": 16384, "N": 4096, "K": 4096},
        # The expert layer: 128 experts, top-8 of 16384 tokens with Zipf load, gate and down projections, forward and backward,
        # groups padded to 128 rows.
        {"name": "experts", "kind": "moe", "T": 16384, "experts": 128, "top_k": 8, "hidden": 2048, "ffn": 768, "pad": 128},
        # The paper's mixed layout: activations in 1D blocks, once along the channels and once along the tokens, at the
        # 1B-class gate projection.
        {"name": "act1d 1B", "kind": "act1d", "T": 8192, "N": 5632, "K": 2048},
        # Layers that hand quantized tensors on: forward and input-gradient products that quantize their own output.
        {"name": "fused 7B", "kind": "fused", "T": 16384, "N": 4096, "K": 4096},
        # The block-size study's 16 x 16 blocks at a 1B-class projection.
        {"name": "block16 1B", "kind": "block16", "T": 8192, "N": 2048, "K": 2048},
    ]


def _spread(rng, lo, hi, step=1):
    """A size between lo and hi, even over its logarithm, rounded to a multiple of step."""
    return max(step, int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) // step * step)


def _size(rng, lo, hi):
    """Half of the sizes are multiples of 128, a quarter of 16, a quarter are whatever comes (mostly odd or ragged)."""
    return _spread(rng, lo, hi, rng.choice([128, 128, 16, 1]))


def draw(rng: random.Random):
    kind = rng.choice(["linear", "linear", "layer", "layer", "microbatch", "quantize", "quantize", "mxfp8", "moe", "act1d", "fused", "block16"])
    if kind == "moe":
        # T * top_k * hidden * ffn stays below the listed expert layer's
        return {"kind": kind, "T": _spread(rng, 256, 16384), "experts": rng.choice([4, 8, 16, 32, 64, 128]), "top_k": rng.choice([1, 2, 4]),
                "hidden": _spread(rng, 256, 2048, 64), "ffn": _spread(rng, 128, 1536, 64), "pad": rng.choice([128, 128, 256])}
    while True:
        T, N, K = _size(rng, 128, 16384), _size(rng, 256, 11008), _size(rng, 256, 11008)
        if T * N * K <= 16384 * 4096 * 4096:
            break
    c = {"kind": kind, "T": T, "N": N, "K": K}
    if kind == "quantize":
        c["stochastic"] = rng.random() < 0.7
    if kind == "fused":
        c["N"], c["K"] = max(32, N // 16 * 16), max(32, K // 16 * 16)   # the fused epilogue takes widths that are multiples of 16
    return c


def _dense_inputs(c, seed, w_dtype=torch.bfloat16):
    T, N, K = c["T"], c["N"], c["K"]
    w = workloads.weights(N, K, 3 * seed, DEVICE).to(w_dtype)
    x = workloads.activations_student_t(T, K, 3 * seed + 1, DEVICE)
    dy = workloads.gradients_rowscaled(T, N, 3 * seed + 2, DEVICE)
    return w, x, dy


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c, "kind": kind, "seed": seed & 0x7FFFFFFF, "ws": binding.alloc_workspace(DEVICE)}
    if kind == "moe":
        cfg = workloads.MoEConfig(experts=c["experts"], hidden=c["hidden"], expert_ffn=c["ffn"], tokens=c["T"], top_k=c["top_k"])
        # the Zipf loads of the case, on other experts for every seed
        counts = np.random.default_rng(seed).permutation(workloads.moe_routing(cfg))
        offs = workloads.padded_row_offsets(counts, c["pad"])
        rows = int(offs[-1])
        valid = torch.zeros(rows, 1, dtype=torch.bool)
        for e, n in enumerate(counts):
            valid[int(offs[e]):int(offs[e]) + int(n)] = True
        valid = valid.to(DEVICE)
        h, f = c["hidden"], c["ffn"]
        for name, n, k, base in (("gate", f, h, 6 * seed), ("down", h, f, 6 * seed + 3)):
            s["w_" + name] = workloads.weights(c["experts"] * n, k, base, DEVICE)
            s["x_" + name] = workloads.activations_student_t(rows, k, base + 1, DEVICE) * valid
            s["dy_" + name] = workloads.gradients_rowscaled(rows, n, base + 2, DEVICE) * valid
        s["offsets"] = torch.from_numpy(offs).to(DEVICE)
        return s
    if kind == "linear":
        w, x, dy = _dense_inputs(c, seed, torch.float32)
        s["w"], s["x"], s["dy"] = w.requires_grad_(), x.requires_grad_(), dy
        return s
    s["w"], s["x"], s["dy"] = _dense_inputs(c, seed)
    if kind == "microbatch":
        s["qw"] = binding.fp4q_quantize2d(s.pop("w"))
        s["dw"] = torch.zeros(c["N"], (c["K"] + 3) // 4 * 4, dtype=torch.float32, device=DEVICE)[:, :c["K"]]
    if kind == "fused":
        # handed on by the neighbouring layers
        s["qw"], s["qx"] = binding.fp4q_quantize2d(s.pop("w")), binding.fp4q_quantize2d(s.pop("x"))
        s["qdy"] = binding.fp4q_quantize2d(s.pop("dy"), mode=binding.ROUND_STOCHASTIC, seed=s["seed"], tensor_id=2)
    if kind == "mxfp8":
        s["wk"] = workloads.weights(c["N"], c["K"], 3 * seed + 7_000_001, DEVICE)
    return s


def run(s):
    c, b, ws = s["case"], binding, s["ws"]
    SR, seed = b.ROUND_STOCHASTIC, s["seed"]
    if s["kind"] == "linear":
        y = autograd.fp4_linear(s["x"], s["w"], seed=seed, tensor_id=1, ws=ws)
        dx, dw = torch.autograd.grad(y, (s["x"], s["w"]), s["dy"])
        return y, dx, dw
    if s["kind"] == "layer":
        qw, qx, qdy = b.fp4q_quantize2d_multi([s["w"], s["x"], s["dy"]], mode=SR, seed=seed)
        return (b.fp4q_gemm_fwd(qx, qw, ws=ws), b.fp4q_gemm_dgrad(qdy, qw, ws=ws), b.fp4q_gemm_wgrad(qdy, qx, ws=ws))
    if s["kind"] == "microbatch":
        qx = b.fp4q_quantize2d(s["x"])
        y = b.fp4q_gemm_fwd(qx, s["qw"], ws=ws)
        qdy = b.fp4q_quantize2d(s["dy"], mode=SR, seed=seed, tensor_id=1)
        dx = b.fp4q_gemm_dgrad(qdy, s["qw"], ws=ws)
        b.fp4q_gemm_wgrad(qdy, qx, out=s["dw"], accumulate=True, ws=ws)
        return y, dx, s["dw"]
    if s["kind"] == "quantize":
        qs = b.fp4q_quantize2d_multi([s["w"], s["x"], s["dy"]], mode=SR if c["stochastic"] else b.ROUND_NEAREST, seed=seed)
        return [(q.q_rm, q.q_t, q.scale) for q in qs]
    if s["kind"] == "mxfp8":
        T, N, K = c["T"], c["N"], c["K"]
        xq, xs = b.fp4q_mxfp8_quantize1d(s["x"])
        wq, wqs = b.fp4q_mxfp8_quantize1d(s["w"])
        wk, wks = b.fp4q_mxfp8_quantize1d(s["wk"])
        q, k = b.fp4q_mxfp8_qk(xq, xs, wq, wqs, wk, wks, T, K, N, ws=ws)
        dyq, dys = b.fp4q_mxfp8_quantize1d(s["dy"])
        wt, wts = b.fp4q_mxfp8_quantize1d_t(s["w"])
        dx = b.fp4q_mxfp8_gemm(dyq, dys, wt, wts, T, K, N, ws=ws)
        dyt, dyts = b.fp4q_mxfp8_quantize1d_t(s["dy"])
        xt, xts = b.fp4q_mxfp8_quantize1d_t(s["x"])
        dw = b.fp4q_mxfp8_gemm(dyt, dyts, xt, xts, N, K, T, dt=b.OUT_F32, ws=ws)
        return q, k, dx, dw
    if s["kind"] == "moe":
        outs, offs, align = [], s["offsets"], c["pad"]
        for name in ("gate", "down"):
            qw, qx = b.fp4q_quantize2d_multi([s["w_" + name], s["x_" + name]])
            qdy = b.fp4q_quantize2d(s["dy_" + name], mode=SR, seed=seed, tensor_id=2)
            outs.append(b.fp4q_gemm_fwd(qx, qw, row_offsets=offs, ws=ws, row_alignment=align))
            outs.append(b.fp4q_gemm_dgrad(qdy, qw, row_offsets=offs, ws=ws, row_alignment=align))
            outs.append(b.fp4q_gemm_wgrad(qdy, qx, row_offsets=offs, ws=ws))
        return outs
    if s["kind"] == "act1d":
        xq, xs = b.fp4q_quantize1d(s["x"])
        xtq, xts = b.fp4q_quantize1d_t(s["x"])
        qw = b.fp4q_quantize2d(s["w"])
        qdy = b.fp4q_quantize2d(s["dy"], mode=SR, seed=seed, tensor_id=1)
        y = b.fp4q_gemm_fwd_act1d(xq, xs, c["T"], qw, ws=ws)
        return y, b.fp4q_gemm_dgrad(qdy, qw, ws=ws), b.fp4q_gemm_wgrad_act1d(qdy, xtq, xts, c["K"], ws=ws)
    if s["kind"] == "fused":
        y = b.fp4q_gemm_fwd_quantized(s["qx"], s["qw"], ws=ws)
        dx = b.fp4q_gemm_dgrad_quantized(s["qdy"], s["qw"], mode=SR, seed=seed, tensor_id=1, ws=ws)
        return [(q.q_rm, q.q_t, q.scale) for q in (y, dx)]
    if s["kind"] == "block16":
        f = b.BLOCK_16
        qw, qx = b.fp4q_quantize2d(s["w"], flags=f), b.fp4q_quantize2d(s["x"], flags=f)
        qdy = b.fp4q_quantize2d(s["dy"], mode=SR, seed=seed, tensor_id=1, flags=f)
        return b.fp4q_gemm_fwd_b16(qx, qw, ws=ws), b.fp4q_gemm_dgrad_b16(qdy, qw, ws=ws), b.fp4q_gemm_wgrad_b16(qdy, qx, ws=ws)
    raise ValueError(s["kind"])


def work(case):
    c, kind = case, case["kind"]
    if kind == "moe":
        cfg = workloads.MoEConfig(experts=c["experts"], hidden=c["hidden"], expert_ffn=c["ffn"], tokens=c["T"], top_k=c["top_k"])
        T, N, K = int(workloads.padded_row_offsets(workloads.moe_routing(cfg), c["pad"])[-1]), c["ffn"], c["hidden"]
        valid, wnk = c["T"] * c["top_k"], c["experts"] * N * K
        # both projections: BF16 weights, activations and gradients in; BF16 outputs and input gradients, FP32 weight gradients out
        return {"bytes": 2 * (2 * wnk + 4 * wnk) + 4 * (2 * T * K + 2 * T * N), "flops": 2 * 6.0 * valid * N * K}
    T, N, K = c["T"], c["N"], c["K"]
    w, x, dy = N * K, T * K, T * N
    code = 1 + 1 / 1024   # bytes per element of a quantized tensor: two payloads and the scales
    flops = 6.0 * T * N * K
    if kind == "linear":
        return {"bytes": 4 * w + 2 * x + 2 * dy + 2 * dy + 2 * x + 4 * w, "flops": flops}
    if kind == "microbatch":   # the weight's codes in both layouts; the running sum is read and written
        return {"bytes": code * w + 2 * x + 2 * dy + 2 * dy + 2 * x + 8 * w, "flops": flops}
    if kind == "quantize":
        return {"bytes": (2 + code) * (w + x + dy), "flops": 0}
    if kind == "mxfp8":
        return {"bytes": 2 * 2 * w + 2 * x + 2 * dy + 2 * 2 * dy + 2 * x + 4 * w, "flops": 8.0 * T * N * K}
    if kind == "fused":        # row-major codes of X and dY, W's in both layouts; two quantized outputs
        return {"bytes": code * w + 0.5 * (x + dy) + code * (dy + x), "flops": 4.0 * T * N * K}
    return {"bytes": 2 * w + 2 * x + 2 * dy + 2 * dy + 2 * x + 4 * w, "flops": flops}   # layer, act1d, block16


def tolerance(case):
    kind = case["kind"]
    if kind == "quantize":
        return "exact"   # codes and scales are defined bit for bit
    if kind == "fused":
        # one sum that falls on the other side of a BF16 rounding boundary can move a code, or a block's scale with its 1024 codes
        return {"rel": 0.0, "differ": 1e-3}
    # Sums of FP4 products are exact in FP32 but for blocks of very different scale, MXFP8 sums differ from 64-bit ones by
    # 2.4e-7; what remains is one rounding to BF16: measured against 64-bit products 1.7e-3 in norm, half a unit (3.9e-3) at most.
    return {"rel": 2e-3, "max": 8e-3}


# ---- the same passes in 64 bits: quantizers and products from their definitions, in plain torch

_E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)


def _exact_bytes(rows, cols, seed, tensor_id):
    """One random byte per element: byte idx % 16 of Philox4x32-10 at counter idx / 16, idx the row-major index."""
    mask = 0xFFFFFFFF
    n = (rows * cols + 15) // 16
    c0 = torch.arange(n, dtype=torch.int64, device=DEVICE)
    c = [c0 & mask, c0 >> 32, torch.full_like(c0, tensor_id), torch.zeros_like(c0)]
    k0, k1 = seed & mask, (seed >> 32) & mask

    def mul(m, x):   # 32 x 32 bits -> (high, low) without leaving int64
        lo, hi = m * (x & 0xFFFF), m * (x >> 16)
        low = lo + ((hi & 0xFFFF) << 16)
        return (hi >> 16) + (low >> 32), low & mask

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    words = torch.stack(c, dim=1)
    b = torch.stack([(words >> (8 * i)) & 0xFF for i in range(4)], dim=2)
    return b.reshape(-1)[:rows * cols].reshape(rows, cols)


def _exact_scale(x, br, bc, top):
    """2^e per element, e the least with top * 2^e >= the largest magnitude of the element's br x bc block."""
    rows, cols = x.shape
    p = torch.nn.functional.pad(x.abs(), (0, -cols % bc, 0, -rows % br))
    m = p.view(p.shape[0] // br, br, p.shape[1] // bc, bc).amax(dim=(1, 3))
    f, e = torch.frexp(m / top)   # m / top = f 2^e, 0.5 <= f < 1
    e = torch.where(f == 0.5, e - 1, e).clamp(min=-127)
    s = torch.ldexp(torch.ones_like(m), torch.where(m == 0, torch.zeros_like(e), e))
    return s.repeat_interleave(br, 0)[:rows].repeat_interleave(bc, 1)[:, :cols]


def _exact_fp4(x, br=32, bc=32, sr=None):
    """x rounded to E2M1 in br x bc blocks, dequantized; sr = (seed, tensor_id): stochastically."""
    x = x.detach().to(torch.bfloat16).double()
    s = _exact_scale(x, br, bc, 6.0)
    v, grid = (x / s).abs(), torch.tensor(_E2M1, dtype=torch.float64, device=DEVICE)
    lo = (torch.searchsorted(grid, v, right=True) - 1).clamp(0, 6)
    pos = (v - grid[lo]) / (grid[lo + 1] - grid[lo])
    if sr is None:
        up = (pos > 0.5) | ((pos == 0.5) & (lo % 2 == 1))
    else:
        up = torch.floor(256 * pos) + _exact_bytes(x.shape[0], x.shape[1], *sr) >= 256
    return torch.copysign(grid[lo + up.long()], x) * s


def _exact_mxfp8(x):
    x = x.detach().double()
    s = _exact_scale(x, 1, 32, 448.0)
    return (x / s).float().to(torch.float8_e4m3fn).double() * s


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("quantize", "fused"):
        return None   # codes and scales
    sr = seed & 0x7FFFFFFF
    if kind == "moe":
        s = prepare(case, seed)
        offs, outs = s["offsets"].tolist(), []
        groups = list(zip(offs[:-1], offs[1:]))
        for name in ("gate", "down"):
            w, x, dy = _exact_fp4(s["w_" + name]), _exact_fp4(s["x_" + name]), _exact_fp4(s["dy_" + name], sr=(sr, 2))
            w = w.view(c["experts"], -1, w.shape[1])
            outs.append(torch.cat([x[a:b] @ w[e].T for e, (a, b) in enumerate(groups)]))
            outs.append(torch.cat([dy[a:b] @ w[e] for e, (a, b) in enumerate(groups)]))
            outs.append(torch.cat([dy[a:b].T @ x[a:b] for a, b in groups]))
        return outs
    w, x, dy = _dense_inputs(c, seed)
    if kind == "mxfp8":
        wk = workloads.weights(c["N"], c["K"], 3 * seed + 7_000_001, DEVICE)
        q = _exact_mxfp8(x)
        return (q @ _exact_mxfp8(w).T, q @ _exact_mxfp8(wk).T, _exact_mxfp8(dy) @ _exact_mxfp8(w.T.contiguous()).T,
                _exact_mxfp8(dy.T.contiguous()) @ _exact_mxfp8(x.T.contiguous()).T)
    if kind == "layer":
        w, x, dy = (_exact_fp4(t, sr=(sr, i)) for i, t in enumerate((w, x, dy)))
        return x @ w.T, dy @ w, dy.T @ x
    if kind == "act1d":
        w, dy = _exact_fp4(w), _exact_fp4(dy, sr=(sr, 1))
        return _exact_fp4(x, 1, 32) @ w.T, dy @ w, dy.T @ _exact_fp4(x, 32, 1)
    b = 16 if kind == "block16" else 32
    w, x, dy = _exact_fp4(w, b, b), _exact_fp4(x, b, b), _exact_fp4(dy, b, b, sr=(sr, 1))
    return x @ w.T, dy @ w, dy.T @ x   # linear, microbatch (its first pass: the sum starts at zero), block16
