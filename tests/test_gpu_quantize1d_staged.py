"""1D-block quantizers of matrices whose rows start anywhere or that are not made of whole tiles, bit for bit against the oracle: both formats,
along the rows and along the columns, on both sides of the sizes at which the staged kernels take over."""
import numpy as np
import pytest
import torch

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
