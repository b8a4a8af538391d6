"""Calls with an explicit stream: everything a call does - allocation, zero fill, workspace, kernels - is in that stream's
order, whatever the current stream is busy with."""
import pytest
import torch

from paper_2607_24953_b200 import binding as b, workloads

pytestmark = pytest.mark.gpu
T, N, K = 384, 320, 256


def _calls():
    x, w, dy = workloads.activations_gauss_outliers(T, K, 1, "cuda"), workloads.weights(N, K, 2, "cuda"), workloads.gradients_rowscaled(T, N, 3, "cuda")
    qx, qw, qd = b.fp4q_quantize2d(x), b.fp4q_quantize2d(w), b.fp4q_quantize2d(dy)
    px, pw, pd = (b.fp4q_quantize2d(t, flags=b.BLOCK_16) for t in (x, w, dy))
    x1, xs1 = b.fp4q_quantize1d(x)
    xt, xts = b.fp4q_quantize1d_t(x)
    x8, xs8 = b.fp4q_mxfp8_quantize1d(x)
    w8, ws8 = b.fp4q_mxfp8_quantize1d(w)
    offs = torch.tensor([0, 128, 384], device="cuda")
    stack = b.fp4q_quantize2d(torch.cat([w, w]))
    fields = lambda q: (q.q_rm, q.q_t, q.scale)
    return {
        "quantize2d": lambda s: fields(b.fp4q_quantize2d(x, stream=s)),
        "quantize2d_multi": lambda s: sum((fields(q) for q in b.fp4q_quantize2d_multi([x, w, dy], stream=s)), ()),
        "quantize1d": lambda s: b.fp4q_quantize1d(x, stream=s),
        "quantize1d_t": lambda s: b.fp4q_quantize1d_t(x, stream=s),
        "mxfp8_quantize1d": lambda s: b.fp4q_mxfp8_quantize1d(x, stream=s),
        "mxfp8_quantize1d_t": lambda s: b.fp4q_mxfp8_quantize1d_t(x, stream=s),
        "gemm_fwd": lambda s: b.fp4q_gemm_fwd(qx, qw, stream=s),
        "gemm_dgrad": lambda s: b.fp4q_gemm_dgrad(qd, qw, stream=s),
        "gemm_wgrad": lambda s: b.fp4q_gemm_wgrad(qd, qx, stream=s),
        "gemm_wgrad added": lambda s: b.fp4q_gemm_wgrad(qd, qx, accumulate=True, stream=s),
        "gemm_fwd grouped": lambda s: b.fp4q_gemm_fwd(qx, stack, row_offsets=offs, stream=s),
        "gemm_fwd_quantized": lambda s: fields(b.fp4q_gemm_fwd_quantized(qx, qw, stream=s)),
        "gemm_dgrad_quantized": lambda s: fields(b.fp4q_gemm_dgrad_quantized(qd, qw, seed=4, stream=s)),
        "gemm_fwd_act1d": lambda s: b.fp4q_gemm_fwd_act1d(x1, xs1, T, qw, stream=s),
        "gemm_wgrad_act1d": lambda s: b.fp4q_gemm_wgrad_act1d(qd, xt, xts, K, accumulate=True, stream=s),
        "gemm_fwd_b16": lambda s: b.fp4q_gemm_fwd_b16(px, pw, stream=s),
        "gemm_wgrad_b16": lambda s: b.fp4q_gemm_wgrad_b16(pd, px, accumulate=True, stream=s),
        "mxfp8_gemm": lambda s: b.fp4q_mxfp8_gemm(x8, xs8, w8, ws8, T, N, K, stream=s),
        "mxfp8_qk": lambda s: b.fp4q_mxfp8_qk(x8, xs8, w8, ws8, w8, ws8, T, K, N, stream=s)}


def _tensors(out):
    return list(out) if isinstance(out, (tuple, list)) else [out]


@pytest.mark.parametrize("by_handle", [False, True])
def test_a_side_stream_does_not_wait_for_the_current_one_nor_share_its_memory(by_handle):
    calls = _calls()
    side = torch.cuda.Stream()
    for name, call in calls.items():
        want = [t.clone() for t in _tensors(call(None))]
        # blocks that the current stream's pool would hand out next, with work on them still to come
        dirty = [torch.empty_like(t) for t in want] + [torch.empty(b.fp4q_workspace_bytes(), dtype=torch.uint8, device="cuda")]
        # everything once before: the first use of a kernel loads it, the first allocation grows the pool, and both may wait
        _on(side, _tensors(call(side)))
        for t in dirty:
            t.view(torch.uint8).fill_(0x5A)
        torch.cuda.synchronize()
        torch.cuda._sleep(400_000_000)                      # about 0.2 s of the current stream
        for t in dirty:
            t.view(torch.uint8).fill_(0x5A)
        pending = torch.cuda.Event()
        pending.record()
        dirty.clear()
        got = _tensors(call(side.cuda_stream if by_handle else side))
        results = [g.cpu() for g in _on(side, got)]         # on the side stream only
        assert not pending.query(), name + ": the current stream was meant to be busy still"
        for g, w in zip(results, want):
            assert torch.equal(g, w.cpu()), name
        torch.cuda.synchronize()
        for g, w in zip(got, want):                         # nothing queued earlier has written to the outputs since
            assert torch.equal(g, w), name


def _on(stream, tensors):
    with torch.cuda.stream(stream):
        copies = [t.cpu() for t in tensors]
    stream.synchronize()
    return copies


def test_results_of_a_side_stream_outlive_their_last_reader():
    # dropped while the current stream still reads them: their memory must not go to the side stream's next call
    x = workloads.activations_gauss_outliers(T, K, 1, "cuda")
    side = torch.cuda.Stream()
    want = b.fp4q_quantize1d(x)[0].clone()
    other = torch.zeros_like(x)
    torch.cuda.synchronize()
    for _ in range(4):
        q, s = b.fp4q_quantize1d(x, stream=side)
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda._sleep(20_000_000)
        late = q.clone()                                    # still to run
        del q, s
        b.fp4q_quantize1d(other, stream=side)               # same sizes: would be handed the same memory
        torch.cuda.synchronize()
        assert torch.equal(late, want)


def test_the_current_streams_own_handle_and_the_default_streams():
    calls = _calls()
    want = [t.clone() for t in _tensors(calls["gemm_fwd"](None))]
    torch.cuda.synchronize()
    for handle in (torch.cuda.current_stream(), torch.cuda.current_stream().cuda_stream, 0, 1, torch.cuda.default_stream()):
        got = _tensors(calls["gemm_fwd"](handle))
        torch.cuda.synchronize()
        assert all(torch.equal(g, w) for g, w in zip(got, want))
