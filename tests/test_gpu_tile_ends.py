"""Where a CTA's stream of tiles ends: the last tile's output leaves through the operand ring, row tiles are numbered in groups with a
smaller last one, and groups of rows are looked up through a copy of their boundaries when these fill more than a cache line."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2607_24953_b200 import binding, workloads
from tests.gpu_util import check_gemm, dequant_from_gpu

pytestmark = pytest.mark.gpu


def operands(*shapes):
    return [binding.fp4q_quantize2d(workloads.activations_student_t(r, c, 7 + i, "cuda")) for i, (r, c) in enumerate(shapes)]


# 18 row tiles of pairs (16 and 2) by 5 column tiles, more than there are pairs, the last column tile 76 wide: pairs with one tile and with
# two, and all products' outputs in both types; one row tile, one CTA; rows that only a pair's first CTA has
@pytest.mark.parametrize("T,N,K", [(4400, 1100, 96), (128, 300, 70), (300, 129, 1000), (1, 1, 1), (4400, 1100, 1400)])
def test_last_tiles(T, N, K):
    ws = binding.alloc_workspace("cuda")
    qx, qw, qdy = operands((T, K), (N, K), (T, N))
    x, w, dy = (dequant_from_gpu(q) for q in (qx, qw, qdy))
    refs = oracle.gemm_fwd(x, w), oracle.gemm_dgrad(dy, w), oracle.gemm_wgrad(dy, x)
    for dt in (binding.OUT_BF16, binding.OUT_F32):
        check_gemm(binding.fp4q_gemm_fwd(qx, qw, dt=dt, ws=ws), refs[0], "fwd")
        check_gemm(binding.fp4q_gemm_dgrad(qdy, qw, dt=dt, ws=ws), refs[1], "dgrad")
        check_gemm(binding.fp4q_gemm_wgrad(qdy, qx, dt=dt, ws=ws), refs[2], "wgrad")
    dw = binding.fp4q_gemm_wgrad(qdy, qx, ws=ws)
    once = dw.clone()
    binding.fp4q_gemm_wgrad(qdy, qx, out=dw, accumulate=True, ws=ws)
    assert torch.equal(dw, 2 * once)
    torch.cuda.synchronize()
    assert binding.fp4q_workspace_status(ws) == 0


# one line of boundaries and more than one, more than the images' place holds, empty groups at both ends and in the middle
@pytest.mark.parametrize("E", [15, 16, 17, 200, 6200])
def test_groups_are_found(E):
    ws = binding.alloc_workspace("cuda")
    rng = np.random.default_rng(E)
    tiles = rng.integers(0, 3, E) if E < 1000 else (rng.random(E) < 0.02).astype(np.int64)
    tiles[[0, E // 2, E - 1]] = 0
    offs = np.concatenate([[0], np.cumsum(128 * tiles)])
    T, N, K = int(offs[-1]), 64, 64
    qx, qw, qdy = operands((T, K), (E * N, K), (T, N))
    x, w, dy = (dequant_from_gpu(q) for q in (qx, qw, qdy))
    d = torch.from_numpy(offs).cuda()
    y, dx = binding.fp4q_gemm_fwd(qx, qw, row_offsets=d, ws=ws), binding.fp4q_gemm_dgrad(qdy, qw, row_offsets=d, ws=ws)
    groups = [(g, slice(int(offs[g]), int(offs[g + 1]))) for g in range(E) if tiles[g]]
    check_gemm(y, np.concatenate([x[s] @ w[g * N:(g + 1) * N].T for g, s in groups]), "fwd")
    check_gemm(dx, np.concatenate([dy[s] @ w[g * N:(g + 1) * N] for g, s in groups]), "dgrad")
    torch.cuda.synchronize()
    assert binding.fp4q_workspace_status(ws) == 0


# Groups on multiples of 128 rows on pairs: two row tiles of a group a pair, the last of an odd number alone; empty groups, one group, more
# groups than tiles, a last tile that is not full, both types of output
@pytest.mark.parametrize("E,rows", [(8, 60), (600, 60), (1, 61), (3, 62)])
def test_paired_rows(E, rows):
    ws = binding.alloc_workspace("cuda")
    rng = np.random.default_rng(E)
    tiles = rng.multinomial(rows, rng.dirichlet(np.full(E, 0.5)))
    offs = np.concatenate([[0], np.cumsum(128 * tiles)])
    T, N, K = int(offs[-1]) - 3, 640, 1056
    qx, qw, qdy = operands((T, K), (E * N, K), (T, N))
    d = torch.from_numpy(offs).cuda()
    full = {dt: (binding.fp4q_gemm_fwd(qx, qw, dt=dt, row_offsets=d, ws=ws), binding.fp4q_gemm_dgrad(qdy, qw, dt=dt, row_offsets=d, ws=ws))
            for dt in (binding.OUT_BF16, binding.OUT_F32)}
    x, dy, w = (torch.from_numpy(dequant_from_gpu(q)) for q in (qx, qdy, qw))
    groups = [(g, slice(int(offs[g]), min(T, int(offs[g + 1])))) for g in range(E) if tiles[g]]
    y = torch.cat([x[s] @ w[g * N:(g + 1) * N].T for g, s in groups]).numpy()
    dx = torch.cat([dy[s] @ w[g * N:(g + 1) * N] for g, s in groups]).numpy()
    for dt in full:
        check_gemm(full[dt][0], y, "fwd")
        check_gemm(full[dt][1], dx, "dgrad")
    torch.cuda.synchronize()
    assert binding.fp4q_workspace_status(ws) == 0


# Weight gradients of experts whose rows do not end with a box of 32: one CTA (up to 128 rows) and pairs, a box within one expert and over several,
# empty experts in every place, both types of output, added to what is there, rows beside the stack untouched
@pytest.mark.parametrize("N", [1, 9, 48, 100, 129, 272, 300])
def test_experts_of_any_number_of_rows(N):
    ws = binding.alloc_workspace("cuda")
    tiles = np.array([0, 2, 1, 0, 0, 3, 1, 5, 0])
    offs = np.concatenate([[0], np.cumsum(128 * tiles)])
    E, T, K = len(tiles), int(offs[-1]), 200
    qx, qdy = operands((T, K), (T, N))
    d = torch.from_numpy(offs).cuda()
    x, dy = (dequant_from_gpu(q) for q in (qx, qdy))
    want = np.concatenate([dy[offs[g]:offs[g + 1]].T @ x[offs[g]:offs[g + 1]] for g in range(E)])
    for dt, dtype in ((binding.OUT_F32, torch.float32), (binding.OUT_BF16, torch.bfloat16)):
        buf = torch.full((E * N + 40, K), 7.0, dtype=dtype, device="cuda")
        check_gemm(binding.fp4q_gemm_wgrad(qdy, qx, out=buf[:E * N], dt=dt, row_offsets=d, ws=ws), want, "wgrad")
        for g in np.flatnonzero(tiles == 0):
            assert not buf[g * N:(g + 1) * N].any()
        assert (buf[E * N:] == 7.0).all()
    dw = torch.zeros(E * N + 40, K, device="cuda")
    for _ in range(2):
        binding.fp4q_gemm_wgrad(qdy, qx, out=dw[:E * N], accumulate=True, row_offsets=d, ws=ws)
    check_gemm(dw[:E * N], 2 * want, "wgrad, added")
    assert not dw[E * N:].any()
    torch.cuda.synchronize()
    assert binding.fp4q_workspace_status(ws) == 0


# A row's last elements, in 16 bytes that the output fills only in part: all kinds, one CTA and pairs, both types; nothing is written beyond them
@pytest.mark.parametrize("T", [1, 128, 300])
@pytest.mark.parametrize("N,K", [(1, 300), (3, 65), (7, 129), (9, 130), (131, 257), (257, 1), (1003, 63), (515, 70)])
def test_outputs_end_with_their_last_column(T, N, K):
    ws = binding.alloc_workspace("cuda")
    x, w, dy = (workloads.activations_student_t(r, c, 7 + i, "cuda") for i, (r, c) in enumerate([(T, K), (N, K), (T, N)]))
    (qx, qw, qdy), (bx, bw, bdy) = ([binding.fp4q_quantize2d(t, flags=flags) for t in (x, w, dy)] for flags in (0, binding.BLOCK_16))
    x1, xt1, x8, w8 = binding.fp4q_quantize1d(x), binding.fp4q_quantize1d_t(x), binding.fp4q_mxfp8_quantize1d(x), binding.fp4q_mxfp8_quantize1d(w)

    def mxfp8(dt, ws, out=None):   # through the C interface, whose output may be any buffer
        out = torch.empty(T, (N + 7) // 8 * 8, dtype=(torch.bfloat16, torch.float32)[dt], device="cuda")[:, :N] if out is None else out
        operands = [v for (q, sc), rows in ((x8, T), (w8, N)) for v in (q.data_ptr(), q.stride(0), sc.data_ptr(), sc.stride(0), rows)]
        assert binding.lib().fp4q_mxfp8_gemm(*operands, K, out.data_ptr(), out.stride(0), dt, ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream) == 0
        return out

    products = [((T, N), False, lambda **k: binding.fp4q_gemm_fwd(qx, qw, **k)), ((T, K), False, lambda **k: binding.fp4q_gemm_dgrad(qdy, qw, **k)),
                ((N, K), True, lambda **k: binding.fp4q_gemm_wgrad(qdy, qx, **k)),
                ((T, N), False, lambda **k: binding.fp4q_gemm_fwd_b16(bx, bw, **k)), ((T, K), False, lambda **k: binding.fp4q_gemm_dgrad_b16(bdy, bw, **k)),
                ((N, K), True, lambda **k: binding.fp4q_gemm_wgrad_b16(bdy, bx, **k)), ((T, N), False, lambda **k: binding.fp4q_gemm_fwd_act1d(*x1, T, qw, **k)),
                ((N, K), True, lambda **k: binding.fp4q_gemm_wgrad_act1d(qdy, *xt1, K, **k)), ((T, N), False, mxfp8)]
    if T % 128 == 0:   # one group
        products.append(((N, K), True, lambda **k: binding.fp4q_gemm_wgrad(qdy, qx, row_offsets=torch.tensor([0, T], device="cuda"), **k)))
    for i, ((rows, cols), adds, product) in enumerate(products):
        for dt, dtype in ((binding.OUT_F32, torch.float32), (binding.OUT_BF16, torch.bfloat16)):
            whole = product(dt=dt, ws=ws)
            buf = torch.full((rows + 3, (cols + 15) // 8 * 8), 7.0, dtype=dtype, device="cuda")
            product(dt=dt, ws=ws, out=buf[:rows, :cols])
            assert torch.equal(buf[:rows, :cols], whole), (i, dtype)
            assert (buf[:rows, cols:] == 7.0).all() and (buf[rows:] == 7.0).all(), (i, dtype)
        if adds:
            once = product(dt=binding.OUT_F32, ws=ws)
            buf = torch.full((rows + 3, (cols + 15) // 8 * 8), -0.0, device="cuda")
            for _ in range(2):
                product(dt=binding.OUT_F32, ws=ws, out=buf[:rows, :cols], accumulate=True)
            assert torch.equal(buf[:rows, :cols], 2 * once), i
            assert torch.signbit(buf[:rows, cols:]).all() and torch.signbit(buf[rows:]).all(), i
    torch.cuda.synchronize()
    assert binding.fp4q_workspace_status(ws) == 0


# An output whose rows are padded may be filled up to 16 bytes, and no further; the binding says so of its own outputs only
def test_padded_outputs():
    ws = binding.alloc_workspace("cuda")
    qx, qw = operands((300, 100), (131, 100))
    want = binding.fp4q_gemm_fwd(qx, qw, ws=ws)
    buf = torch.full((300, 160), 7.0, dtype=torch.bfloat16, device="cuda")
    cx, cw = qx.c_struct(), qw.c_struct()
    assert binding.lib().fp4q_gemm_fwd(ctypes.byref(cx), ctypes.byref(cw), buf.data_ptr(), 160, 0x100 | binding.OUT_BF16, None, ws.data_ptr(), ws.numel(),
                                       torch.cuda.current_stream().cuda_stream) == 0
    assert torch.equal(buf[:, :131], want) and (buf[:, 136:] == 7.0).all()
    for dt in (0x100, 0x101, 2, 0xFF):
        with pytest.raises(binding.Fp4qError):
            binding.fp4q_gemm_fwd(qx, qw, dt=dt, ws=ws)


# 81 tiles of 43 and of 44 stages: both sides of the line (48 stages for each of 74 pairs) from which on a dense product runs with a
# watcher between the loads and the MMAs; and that every role leaves there, too, when a load that it waits for never arrives
@pytest.mark.parametrize("K", [43 * 256, 44 * 256])
def test_short_and_long_products(K):
    ws = binding.alloc_workspace("cuda")
    qx, qw, qdy = operands((2304, K), (2304, K), (2304, 2304))
    binding.fp4q_workspace_set_wait_limit(ws, 1 << 12)
    binding.fp4q_debug_withhold_load(ws, 5)
    binding.fp4q_gemm_fwd(qx, qw, ws=ws)
    torch.cuda.synchronize()
    assert binding.fp4q_workspace_status(ws) == 7
    binding.fp4q_debug_withhold_load(ws, 0)
    binding.fp4q_workspace_set_wait_limit(ws, 0)
    rows = slice(5, None, 97)
    x, w, dy = (dequant_from_gpu(q) for q in (qx, qw, qdy))
    check_gemm(binding.fp4q_gemm_fwd(qx, qw, ws=ws)[rows], oracle.gemm_fwd(x[rows], w), "fwd")
    check_gemm(binding.fp4q_gemm_dgrad(qdy, qw, ws=ws)[rows], oracle.gemm_dgrad(dy[rows], w), "dgrad")
    check_gemm(binding.fp4q_gemm_wgrad(qdy, qx, ws=ws)[rows], oracle.gemm_wgrad(np.ascontiguousarray(dy[:, rows]), x), "wgrad")
    torch.cuda.synchronize()
    assert binding.fp4q_workspace_status(ws) == 0
