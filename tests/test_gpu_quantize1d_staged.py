"""1D-block quantizers of matrices whose rows start anywhere or that are not made of whole tiles, bit for bit against the oracle: both formats,
along the rows and along the columns, on both sides of the sizes at which the staged kernels take over."""
import numpy as np
import pytest
import torch
from torch.profiler import ProfilerActivity, profile

import oracle
from paper_2607_24953_b200 import binding, workloads

pytestmark = pytest.mark.gpu


def matrix(rows, cols, pitch, start):
    """A view that starts anywhere, between other values, with non-finite entries in some blocks."""
    buf = torch.full((start + rows * pitch + 8,), 3.0e38, dtype=torch.bfloat16, device="cuda")
    x = buf.as_strided((rows, cols), (pitch, 1), start)
    x.copy_(workloads.activations_student_t(rows, cols, rows + cols, "cuda"))
    g = torch.Generator().manual_seed(rows)
    for value in (float("inf"), -float("inf"), float("nan")):
        for _ in range(3):
            x[int(torch.randint(rows, (1,), generator=g)), int(torch.randint(cols, (1,), generator=g))] = value
    return x


# tiles' edges in both directions, one row, one column, rows on words, on 16 and 32 bytes and on none; from 1.5 million elements on along the rows,
# from 6 million on for rows on words along the columns
@pytest.mark.parametrize("rows,cols,pitch,start", [(1, 1, 1, 1), (31, 33, 35, 0), (33, 129, 129, 3), (128, 128, 129, 0), (129, 257, 257, 5), (130, 1, 7, 1), (1, 1000, 1001, 0),
                                                    (300, 777, 777, 0), (96, 200, 202, 2), (1201, 1311, 1311, 0), (1300, 1216, 1217, 1), (2500, 2502, 2502, 0), (2500, 2512, 2512, 0)])
def test_any_rows(rows, cols, pitch, start):
    x = matrix(rows, cols, pitch, start)
    bits = workloads.bf16_bits(x.contiguous())
    cases = [(binding.fp4q_quantize1d, oracle.quantize1d, 2, cols), (binding.fp4q_quantize1d_t, oracle.quantize1d_t, 2, rows),
             (binding.fp4q_mxfp8_quantize1d, oracle.mxfp8_quantize1d, 1, cols), (binding.fp4q_mxfp8_quantize1d_t, oracle.mxfp8_quantize1d_t, 1, rows)]
    for quantize, reference, per_byte, length in cases:
        q, s = quantize(x)
        want_q, want_s = reference(bits)
        got_q, n = q.cpu().numpy(), (length + per_byte - 1) // per_byte
        assert np.array_equal(s.cpu().numpy()[:, :(length + 31) // 32], want_s), quantize.__name__
        assert np.array_equal(got_q[:, :n], want_q), quantize.__name__
        assert not got_q[:, n:(length + 31) // 32 * 32 // per_byte].any(), quantize.__name__   # block padding


# Few rows or few columns, where tiles are mostly empty: the element-wise kernels whatever the number of elements, along the rows below 20 rows or 360
# columns, along the columns below 16 rows or 8 columns or in more than 400 tiles that are less than a quarter full; rows on words in tiles that are not
# nearly full; and what goes through tiles just beside these
@pytest.mark.parametrize("rows,cols,pitch,start", [(1, 1600001, 1600001, 1), (19, 83001, 83001, 0), (20, 83001, 83001, 3), (33, 50001, 50001, 0), (15, 60001, 60001, 0),
                                                    (16, 60001, 60001, 0), (16, 9001, 9001, 1), (32, 60001, 60001, 0), (60001, 33, 33, 1), (200001, 17, 17, 0), (4400, 359, 359, 0),
                                                    (4400, 361, 361, 0), (70001, 7, 7, 0), (4001, 8, 9, 0), (33, 1100002, 1100002, 0)])
def test_few_rows_or_columns(rows, cols, pitch, start):
    test_any_rows(rows, cols, pitch, start)


def kernels(call):
    call()
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        call()
        torch.cuda.synchronize()
    return " ".join(e.key for e in p.key_averages())


# one row, a few, narrow ones: as many tiles as a matrix of 128 times the elements has; and what is made of full tiles
@pytest.mark.parametrize("rows,cols,along_rows,along_columns", [(1, 2000001, False, False), (16, 151937, False, False), (60000, 33, False, True), (600001, 3, False, False),
                                                                (33, 60001, True, True), (1999, 1003, True, True)])
def test_work_is_counted_in_tiles(rows, cols, along_rows, along_columns):
    x = torch.zeros(rows * cols + 1, dtype=torch.bfloat16, device="cuda")[1:].view(rows, cols)
    for quantize, staged in ((binding.fp4q_quantize1d, along_rows), (binding.fp4q_mxfp8_quantize1d, along_rows),
                             (binding.fp4q_quantize1d_t, along_columns), (binding.fp4q_mxfp8_quantize1d_t, along_columns)):
        names = kernels(lambda: quantize(x))
        assert "quantize1d" in names and ("staged" in names) == staged, (quantize.__name__, names)
