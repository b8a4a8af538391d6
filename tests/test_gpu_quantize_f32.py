"""FP32 sources: the result is that of the BF16 quantizer on a BF16 copy, bit for bit."""
import ctypes

import pytest
import torch

from paper_2607_24953_b200 import binding

pytestmark = pytest.mark.gpu


def quantize_f32(xs, is_f32, mode, seed):
    L, jobs, outs, keep = binding.lib(), (binding._CQuantJob * len(xs))(), [], []
    for j, x in enumerate(xs):
        outs.append(binding.alloc_qtensor(x.shape[0], x.shape[1], "cuda"))
        keep.append(outs[-1].c_struct())
        jobs[j] = binding._CQuantJob(x.data_ptr(), x.shape[0], x.shape[1], x.stride(0), ctypes.pointer(keep[-1]), j, 0)
    st = L.fp4q_quantize2d_multi_f32(jobs, bytes(is_f32), len(xs), mode, seed, torch.cuda.current_stream().cuda_stream)
    return st, outs


# whole tiles, remainders of every kind, rows on 32 and on 16 bytes, a pitch
@pytest.mark.parametrize("rows,cols,pitch", [(128, 128, 128), (1, 4, 4), (33, 100, 100), (256, 264, 264), (130, 1004, 1004), (97, 61, 64), (300, 120, 136), (513, 384, 388)])
@pytest.mark.parametrize("mode", [binding.ROUND_NEAREST, binding.ROUND_STOCHASTIC])
def test_fp32_sources_match_their_bf16_copies(rows, cols, pitch, mode):
    g = torch.Generator(device="cuda").manual_seed(rows + cols)
    x = (torch.randn(rows, pitch, generator=g, device="cuda") * torch.exp2(torch.randint(-20, 20, (rows, 1), generator=g, device="cuda").float()))[:, :cols]
    if rows > 64:   # what BF16 rounds to infinity, NaN, subnormals, ties, and a block of zeros
        x[40, 1], x[41, 2], x[42, 3], x[43, 4] = 3.4e38, float("nan"), -float("inf"), 1e-40
        x[50, :cols // 2] = 1.00390625
        x[64:96, :32] = 0.0
    y = x.to(torch.bfloat16).contiguous()
    b = torch.randn(70, 40, generator=g, device="cuda").to(torch.bfloat16)
    st, (qb, qx) = quantize_f32([b, x], [0, 1], mode, 11)
    assert st == 0
    for got, want in ((qx, binding.fp4q_quantize2d(y, mode=mode, seed=11, tensor_id=1)), (qb, binding.fp4q_quantize2d(b, mode=mode, seed=11, tensor_id=0))):
        r, c = got.rows, got.cols
        assert torch.equal(got.scale, want.scale)
        assert torch.equal(got.q_rm[:, :(c + 31) // 32 * 16], want.q_rm[:, :(c + 31) // 32 * 16])
        assert torch.equal(got.q_t[:, :(r + 31) // 32 * 16], want.q_t[:, :(r + 31) // 32 * 16])


def test_unaligned_fp32_sources_are_refused():
    x = torch.zeros(64, 70, device="cuda")
    assert quantize_f32([x[:, 1:65]], [1], 0, 0)[0] == 3       # the address
    assert quantize_f32([x], [1], 0, 0)[0] == 3                # the pitch


# Rows on 16 but not on 32 bytes, by the address or by the pitch: whole tiles and tiles at every edge.
@pytest.mark.parametrize("rows,cols,pitch,start", [(128, 128, 128, 4), (256, 256, 260, 0), (257, 260, 260, 4), (384, 272, 276, 12), (160, 132, 132, 0), (129, 1028, 1028, 0)])
@pytest.mark.parametrize("mode", [binding.ROUND_NEAREST, binding.ROUND_STOCHASTIC])
def test_rows_on_16_bytes_match_their_bf16_copies(rows, cols, pitch, start, mode):
    g = torch.Generator(device="cuda").manual_seed(rows * cols + start)
    buf = torch.randn(start + rows * pitch, generator=g, device="cuda") * torch.exp2(torch.randint(-8, 9, (start + rows * pitch,), generator=g, device="cuda").float())
    x = buf[start:].view(rows, pitch)[:, :cols]
    x[rows - 1, cols - 1], x[0, cols // 2], x[rows // 2, 0] = 3.4e38, float("nan"), float("inf")
    st, (q,) = quantize_f32([x], [1], mode, 5)
    assert st == 0
    want = binding.fp4q_quantize2d(x.to(torch.bfloat16).contiguous(), mode=mode, seed=5, tensor_id=0)
    assert torch.equal(q.scale, want.scale)
    assert torch.equal(q.q_rm[:, :(cols + 31) // 32 * 16], want.q_rm[:, :(cols + 31) // 32 * 16])
    assert torch.equal(q.q_t[:, :(rows + 31) // 32 * 16], want.q_t[:, :(rows + 31) // 32 * 16])
