"""The scale matrices of 2D-block tensors at any pitch and start: the products read them as whole words, as pairs of words shifted
into place, or byte by byte at the matrix's ends, by their alignment and the contraction's length.  Gaps between the rows hold
0xFF, UE8M0's NaN, so that a byte that does not belong to the tensor shows."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2607_24953_b200 import binding, workloads
from tests.gpu_util import check_gemm, dequant_from_gpu

pytestmark = pytest.mark.gpu


def elsewhere(q, gap, start):
    """q with its scale matrix `start` bytes into a buffer, its rows `gap` bytes further apart."""
    rows, cols = q.scale.shape
    buf = torch.full((start + rows * (cols + gap),), 0xFF, dtype=torch.uint8, device="cuda")
    scale = buf.as_strided((rows, cols), (cols + gap, 1), start)
    scale.copy_(q.scale)
    return dataclasses.replace(q, scale=scale)


# contractions of 1, 2, 5, 10, 11, 12, 22, 31 and 33 chunks of 128 in one of the three products, row tiles at the tile's edge and beyond,
# second CTAs of a pair that have no rows
@pytest.mark.parametrize("T,N,K", [(100, 70, 200), (300, 777, 1234), (161, 1311, 2731), (257, 640, 1280), (520, 1400, 4200), (128, 256, 3968), (1500, 300, 70)])
def test_products_do_not_depend_on_where_the_scales_lie(T, N, K):
    g = torch.Generator(device="cuda").manual_seed(T + N + K)
    scales = torch.exp2(torch.randint(-6, 7, (3,), generator=g, device="cuda").float())
    x, w, dy = ((torch.randn(r, c, generator=g, device="cuda") * s * torch.exp2(torch.randint(-4, 5, (r, 1), generator=g, device="cuda").float())).to(torch.bfloat16)
                for (r, c), s in zip(((T, K), (N, K), (T, N)), scales))
    qx, qw, qdy = (binding.fp4q_quantize2d(t) for t in (x, w, dy))
    ws = binding.alloc_workspace("cuda")

    def products(x, w, dy):
        return [binding.fp4q_gemm_fwd(x, w, dt=binding.OUT_F32, ws=ws), binding.fp4q_gemm_dgrad(dy, w, dt=binding.OUT_F32, ws=ws),
                binding.fp4q_gemm_wgrad(dy, x, ws=ws)]

    plain = products(qx, qw, qdy)
    xd, wd, dyd = (dequant_from_gpu(q) for q in (qx, qw, qdy))
    for got, ref, what in zip(plain, (oracle.gemm_fwd(xd, wd), oracle.gemm_dgrad(dyd, wd), oracle.gemm_wgrad(dyd, xd)), ("fwd", "dgrad", "wgrad")):
        check_gemm(got, ref, what)
    for gap, start in ((0, 1), (1, 0), (2, 3), (4 - qx.scale.shape[1] % 4, 4), (7, 2)):
        for got, ref, what in zip(products(*(elsewhere(q, gap, start) for q in (qx, qw, qdy))), plain, ("fwd", "dgrad", "wgrad")):
            assert torch.equal(got, ref), (what, gap, start)   # the same operands and order of sums
    torch.cuda.synchronize()
    assert binding.fp4q_workspace_status(ws) == 0


# Units of the builder (32 chunks of 128) that are full, in each of the three products, and units of every other length up to that.
@pytest.mark.parametrize("T,N,K", [(70, 100, 4100), (100, 4100, 70), (4100, 100, 70), (40, 3970, 3970), (3970, 130, 40), (1500, 1700, 1900), (2200, 2500, 2800), (3100, 3400, 3700)])
def test_units_of_every_length(T, N, K):
    test_products_do_not_depend_on_where_the_scales_lie(T, N, K)


# Grouped products: every group's scales start somewhere else in the matrix.  Contractions of 12, 2, 33 and 34 chunks in the forward product,
# of 1, 32 and 33 in the input gradient, and groups of up to 34 chunks, empty ones among them, in the weight gradient.
@pytest.mark.parametrize("counts,N,K", [((4224, 0, 1400, 1), 96, 100), ((130, 0, 300), 128, 1440), ((129, 1, 0, 260), 64, 4250), ((200, 300), 4096, 160), ((1, 500, 3968), 4160, 100)])
@pytest.mark.parametrize("alignment", [128, 256])
def test_grouped_products_do_not_depend_on_where_the_scales_lie(counts, N, K, alignment):
    counts = np.array(counts)
    offs = workloads.padded_row_offsets(counts, alignment)
    T, E = int(offs[-1]), len(counts)
    g = torch.Generator(device="cuda").manual_seed(T + N + K)
    x, dy = (workloads.zero_padding_rows((torch.randn(T, c, generator=g, device="cuda") * torch.exp2(torch.randint(-4, 5, (T, 1), generator=g, device="cuda").float())).to(torch.bfloat16),
                                         counts, offs) for c in (K, N))
    w = (torch.randn(E * N, K, generator=g, device="cuda") * torch.exp2(torch.randint(-4, 5, (E * N, 1), generator=g, device="cuda").float())).to(torch.bfloat16)
    qx, qw, qdy = (binding.fp4q_quantize2d(t) for t in (x, w, dy))
    ws, d_offs = binding.alloc_workspace("cuda"), torch.from_numpy(offs).cuda()
    dgrad = N % 64 == 0   # a group's contraction ends between two instructions' shares otherwise, and is refused

    def products(x, w, dy):
        rows = dict(dt=binding.OUT_F32, row_offsets=d_offs, ws=ws, row_alignment=alignment)
        dw = binding.fp4q_gemm_wgrad(dy, x, row_offsets=d_offs, ws=ws)
        return [binding.fp4q_gemm_fwd(x, w, **rows), dw] + ([binding.fp4q_gemm_dgrad(dy, w, **rows)] if dgrad else [])

    plain = products(qx, qw, qdy)
    xd, wd, dyd = (dequant_from_gpu(q) for q in (qx, qw, qdy))
    check_gemm(plain[0], oracle.grouped(oracle.gemm_fwd, xd, wd, offs), "fwd")
    if dgrad:
        check_gemm(plain[2], oracle.grouped(oracle.gemm_dgrad, dyd, wd, offs), "dgrad")
    ref = oracle.grouped_wgrad(dyd, xd, offs)
    for e in np.flatnonzero(counts):   # by expert: a small one is not hidden by a large one
        check_gemm(plain[1][e * N:(e + 1) * N], ref[e * N:(e + 1) * N], "wgrad of expert %d" % e)
    for gap, start in ((0, 1), (1, 0), (2, 3), (4 - qx.scale.shape[1] % 4, 4), (7, 2)):
        for got, ref, what in zip(products(*(elsewhere(q, gap, start) for q in (qx, qw, qdy))), plain, ("fwd", "wgrad", "dgrad")):
            assert torch.equal(got, ref), (what, gap, start)
    torch.cuda.synchronize()
    assert binding.fp4q_workspace_status(ws) == 0


def moved(scale, gap, start):
    """A scale matrix `start` bytes into a buffer, its rows `gap` bytes further apart."""
    rows, cols = scale.shape
    buf = torch.full((start + rows * (cols + gap),), 0xFF, dtype=torch.uint8, device="cuda")
    view = buf.as_strided((rows, cols), (cols + gap, 1), start)
    view.copy_(scale)
    return view


# The per-row kinds fetch rows on 16 bytes as they are and others word by word: rows of 1, 3, 7, 8, 16, 17 and 86 blocks (twice that in 16 x 16
# blocks), one unit and several, tiles with one row, with rows at the tile's edge and beyond, one CTA and pairs.
@pytest.mark.parametrize("T,N,K", [(1, 1, 32), (100, 70, 200), (128, 256, 256), (300, 777, 1234), (161, 1311, 2731), (257, 512, 544), (512, 1024, 512), (700, 96, 2080)])
def test_per_row_products_do_not_depend_on_where_the_scales_lie(T, N, K):
    x, w, dy = (workloads.activations_student_t(r, c, i, "cuda") for i, (r, c) in enumerate(((T, K), (N, K), (T, N))))
    ws = binding.alloc_workspace("cuda")
    qw, qdy, q16 = binding.fp4q_quantize2d(w), binding.fp4q_quantize2d(dy), [binding.fp4q_quantize2d(t, flags=binding.BLOCK_16) for t in (x, w, dy)]
    (xq, xs), (xtq, xts) = binding.fp4q_quantize1d(x), binding.fp4q_quantize1d_t(x)
    (mq, ms), (nq, ns) = binding.fp4q_mxfp8_quantize1d(x), binding.fp4q_mxfp8_quantize1d(w)

    def products(move, move_q):
        w2, dy2, (x16, w16, dy16) = move_q(qw), move_q(qdy), [move_q(q) for q in q16]
        return [binding.fp4q_gemm_fwd_act1d(xq, move(xs), T, w2, dt=binding.OUT_F32, ws=ws), binding.fp4q_gemm_wgrad_act1d(dy2, xtq, move(xts), K, ws=ws),
                binding.fp4q_gemm_fwd_b16(x16, w16, dt=binding.OUT_F32, ws=ws), binding.fp4q_gemm_dgrad_b16(dy16, w16, dt=binding.OUT_F32, ws=ws),
                binding.fp4q_gemm_wgrad_b16(dy16, x16, ws=ws), binding.fp4q_mxfp8_gemm(mq, move(ms), nq, move(ns), T, N, K, dt=binding.OUT_F32, ws=ws)]

    plain = products(lambda s: s, lambda q: q)
    xd = {k: torch.from_numpy(v).cuda() for k, v in dict(
        x1=oracle.dequantize1d(xq.cpu().numpy()[:, :(K + 1) // 2].copy(), xs.cpu().numpy()[:, :(K + 31) // 32].copy(), T, K),
        w=dequant_from_gpu(qw), dy=dequant_from_gpu(qdy)).items()}
    check_gemm(plain[0], (xd["x1"] @ xd["w"].T).cpu().numpy(), "1D forward")
    for gap, start in ((0, 0), (0, 1), (1, 0), (2, 3), (16 - xs.shape[1] % 16, 0), (16 - xs.shape[1] % 16, 4), (7, 2)):
        got = products(lambda s: moved(s, gap, start), lambda q: dataclasses.replace(q, scale=moved(q.scale, gap, start)))
        for i, (a, b) in enumerate(zip(got, plain)):
            assert torch.equal(a, b), (i, gap, start)   # the same operands and order of sums
    torch.cuda.synchronize()
    assert binding.fp4q_workspace_status(ws) == 0
