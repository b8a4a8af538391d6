"""Short kernels start beside their predecessor's end (programmatic dependent launches).  Streams must keep their order all
the same: chains of calls on reused buffers with new data every pass, without any synchronisation, against the same
calls with a synchronisation after each."""
import glob
import os
import re

import pytest
import torch

from paper_2607_24953_b200 import binding as b, workloads

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_24953_b200", "csrc")
SR = b.ROUND_STOCHASTIC


def test_kernels_that_start_early_read_through_the_coherent_path():
    # ld.global.nc and __ldg are for memory that nothing writes during the kernel; these kernels begin before their
    # predecessor has written their inputs
    sources = glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    assert sources
    for path in sources:
        code = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.search(r"__ldg\s*\(|\.global\.nc|ld\.nc\b|__restrict__", code), path


def _randn(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda").to(torch.bfloat16)


class Layers:
    """Two layers' worth of calls of every kind on buffers that every pass reuses."""

    def __init__(self, T, N, K):
        self.T, self.N, self.K, self.ws = T, N, K, b.alloc_workspace("cuda")
        self.x, self.dy = (torch.empty(T, n, device="cuda", dtype=torch.bfloat16) for n in (K, N))
        self.w = workloads.weights(N, K, 5, "cuda")
        self.qw, self.qw16 = b.fp4q_quantize2d(self.w), b.fp4q_quantize2d(self.w, flags=b.BLOCK_16)
        self.wq, self.wsc = b.fp4q_mxfp8_quantize1d(self.w)
        self.qx, self.qdy = b.alloc_qtensor(T, K, "cuda"), b.alloc_qtensor(T, N, "cuda")
        self.qx16 = b.alloc_qtensor(T, K, "cuda", True, 16)
        self.y = torch.empty(T, (N + 7) // 8 * 8, device="cuda", dtype=torch.bfloat16)[:, :N]
        self.qy = b.alloc_qtensor(T, N, "cuda")
        self.dx = torch.empty(T, (K + 7) // 8 * 8, device="cuda", dtype=torch.bfloat16)[:, :K]
        self.dw = torch.zeros(N, (K + 3) // 4 * 4, device="cuda")[:, :K]

    def run(self, i, xs, dys, after):
        out = []
        for call in (
                lambda: (self.x.copy_(xs[i % len(xs)]), self.dy.copy_(dys[i % len(dys)])),
                lambda: b.fp4q_quantize2d(self.x, self.qx, mode=SR, seed=i, tensor_id=1),
                lambda: b.fp4q_gemm_fwd(self.qx, self.qw, out=self.y, ws=self.ws),
                lambda: b.fp4q_quantize2d(self.y, self.qy),                                  # reads what the product just wrote
                lambda: b.fp4q_gemm_dgrad(self.qy, self.qw, out=self.dx, ws=self.ws),
                lambda: out.append(self.dx.clone()),
                lambda: b.fp4q_quantize2d_multi([self.dx, self.dy], [self.qx, self.qdy], mode=SR, seed=i),   # overwrites qx, reads dx
                lambda: b.fp4q_gemm_wgrad(self.qdy, self.qx, out=self.dw, accumulate=True, ws=self.ws),
                lambda: self.dx.zero_(),                                                     # an input overwritten right behind its reader
                lambda: b.fp4q_quantize2d(self.dy, self.qdy),
                lambda: out.append(b.fp4q_gemm_dgrad(self.qdy, self.qw, dt=b.OUT_F32, ws=self.ws)),
                lambda: self.dy.zero_(),
                lambda: out.extend(b.fp4q_mxfp8_quantize1d(self.x)),
                lambda: out.append(b.fp4q_mxfp8_gemm(out[-2], out[-1], self.wq, self.wsc, self.T, self.N, self.K, ws=self.ws)),
                lambda: out.extend(b.fp4q_quantize1d(self.x)),
                lambda: out.append(b.fp4q_gemm_fwd_act1d(out[-2], out[-1], self.T, self.qw, ws=self.ws)),
                lambda: b.fp4q_quantize2d(self.x, self.qx16, flags=b.BLOCK_16),
                lambda: out.append(b.fp4q_gemm_fwd_b16(self.qx16, self.qw16, ws=self.ws)),
                lambda: self.x.zero_(),
                lambda: out.append(self.dw.clone())):
            call()
            after()
        return out


@pytest.mark.gpu
@pytest.mark.parametrize("T,N,K", [(128, 256, 256), (300, 520, 544), (512, 512, 1024), (1999, 1003, 731), (4096, 2048, 512)])
def test_chains_without_synchronisation_match_synchronised_ones(T, N, K):
    xs, dys = [_randn(i, T, K) for i in range(3)], [_randn(10 + i, T, N) for i in range(4)]
    passes = 24 if T <= 512 else 6
    plain, ref = Layers(T, N, K), Layers(T, N, K)
    torch.cuda.synchronize()
    got = [plain.run(i, xs, dys, lambda: None) for i in range(passes)]
    want = [ref.run(i, xs, dys, torch.cuda.synchronize) for i in range(passes)]
    torch.cuda.synchronize()
    assert b.fp4q_workspace_status(plain.ws) == 0
    for i, (g, w) in enumerate(zip(got, want)):
        for j, (a, c) in enumerate(zip(g, w)):
            assert torch.equal(a, c), (i, j)


@pytest.mark.gpu
def test_short_and_long_launches_around_a_multi_tensor_call():
    # a long quantizer, a short one, a multi-tensor call whose tensors are short and long in turn, a product of the first
    # and the last of them, and an overwrite of everything read
    big, small, mid = (_randn(k, *s) for k, s in ((1, (8192, 2048)), (2, (256, 2048)), (3, (1024, 2048))))
    ws = b.alloc_workspace("cuda")

    def chain(after):
        out = []
        for i in range(8):
            a, c, d = (t * (1 + i) for t in (big, small, mid))
            q = [b.alloc_qtensor(t.shape[0], t.shape[1], "cuda") for t in (a, c, d)]
            for call in (lambda: b.fp4q_quantize2d(a, q[0], mode=SR, seed=i), lambda: b.fp4q_quantize2d(c, q[1], mode=SR, seed=i),
                         lambda: b.fp4q_quantize2d_multi([c, a, d, c], [q[1], q[0], q[2], b.alloc_qtensor(256, 2048, "cuda")], mode=SR, seed=i),
                         lambda: out.append(b.fp4q_gemm_fwd(q[0], q[1], ws=ws)), lambda: out.append(b.fp4q_gemm_fwd(q[2], q[1], ws=ws)),
                         lambda: [t.zero_() for t in (a, c, d)], lambda: out.append(b.fp4q_gemm_dgrad(b.fp4q_quantize2d(c[:, :1024]), q[2], ws=ws))):
                call()
                after()
        return out

    got = chain(lambda: None)
    want = chain(torch.cuda.synchronize)
    torch.cuda.synchronize()
    assert all(torch.equal(g, w) for g, w in zip(got, want))


@pytest.mark.gpu
@pytest.mark.parametrize("T,N,K", [(128, 256, 256), (1024, 1024, 512)])
def test_a_captured_graph_with_a_fork_and_a_join(T, N, K):
    x, dy, w = _randn(1, T, K), _randn(2, T, N), workloads.weights(N, K, 3, "cuda")
    ws, ws2 = b.alloc_workspace("cuda"), b.alloc_workspace("cuda")
    side = torch.cuda.Stream()

    def body():
        qx, qw, qd = b.fp4q_quantize2d_multi([x, w, dy], mode=SR, seed=9)
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            dx = b.fp4q_gemm_dgrad(qd, qw, ws=ws2)
            qdx = b.fp4q_quantize2d(dx)
        y = b.fp4q_gemm_fwd(qx, qw, ws=ws)
        dw = b.fp4q_gemm_wgrad(qd, qx, ws=ws)
        torch.cuda.current_stream().wait_stream(side)
        return y, dw, b.fp4q_gemm_fwd(qdx, qw, ws=ws), qw.q_rm, qdx.q_rm

    eager = [t.clone() for t in body()]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured = body()
    for scale in (1.0, 0.5, 1.0):      # new data in the captured buffers each time
        x.mul_(0).add_(_randn(1, T, K) * scale)
        for _ in range(3):
            graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(c, e) for c, e in zip(captured, eager))
    assert b.fp4q_workspace_status(ws) == 0 and b.fp4q_workspace_status(ws2) == 0
