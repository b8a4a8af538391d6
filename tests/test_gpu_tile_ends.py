"""Where a CTA's stream of tiles ends: the last tile's output leaves through the operand ring, and row tiles are numbered in groups
with a smaller last one."""
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
