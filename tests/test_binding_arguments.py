"""Arguments of the binding as programs hand them over: whole numbers from NumPy and torch.  An empty list of tensors runs
the whole call without a device, so the argument handling is tested here."""
import numpy as np
import pytest
import torch

from paper_2607_24953_b200 import autograd, binding


@pytest.mark.parametrize("number", [np.int64(3), np.int32(3), np.uint8(3), torch.tensor(3), True, -1, 2 ** 70])
def test_whole_numbers_of_any_type_are_taken(number):
    binding.fp4q_quantize2d_multi([], seed=number, stream=0)
    binding.fp4q_quantize2d_multi([], flags=number, stream=0)


@pytest.mark.parametrize("mode", [np.int64(1), torch.tensor(1), np.uint32(0)])
def test_rounding_modes_of_any_whole_number_type(mode):
    binding.fp4q_quantize2d_multi([], mode=mode, stream=0)


@pytest.mark.parametrize("what", ["seed", "mode", "flags"])
@pytest.mark.parametrize("value", [1.5, "3", None])
def test_other_things_than_whole_numbers_are_refused(what, value):
    with pytest.raises(TypeError):
        binding.fp4q_quantize2d_multi([], stream=0, **{what: value})


def test_a_linear_layer_of_no_inputs_is_refused():
    with pytest.raises(RuntimeError, match="reshape"):
        autograd.fp4_linear(torch.empty(3, 0), torch.empty(4, 0), ws=torch.empty(0))


def test_lists_of_tensors_need_a_length():
    with pytest.raises(TypeError):
        binding.fp4q_quantize2d_multi((t for t in ()), stream=0)
    assert binding.fp4q_quantize2d_multi((), outs=[], stream=0) == []
    with pytest.raises(ValueError):       # a surplus output of the wrong granularity is refused like any other
        binding.fp4q_quantize2d_multi([], outs=[binding.alloc_qtensor(32, 32, "cpu", True, 16)], stream=0)


class _Meddling:
    """A QTensor whose first reader empties the lists that the call was given."""

    def __init__(self, q, lists):
        self._q, self._lists = q, lists

    def __getattr__(self, name):
        for l in self._lists:
            l.clear()
        return getattr(self._q, name)


@pytest.mark.gpu
def test_lists_may_change_while_the_call_runs():
    want = [torch.randn(96, 64, device="cuda").to(torch.bfloat16) for _ in range(3)]
    ref = binding.fp4q_quantize2d_multi(want)
    got = [binding.alloc_qtensor(96, 64, "cuda") for _ in want]
    xs, ids, outs = [t.clone() for t in want], [0, 1, 2], []
    outs += [_Meddling(got[0], [xs, outs])] + got[1:]
    assert binding.fp4q_quantize2d_multi(xs, outs, tensor_ids=ids) is outs and not xs
    for a, c in zip(ref, got):
        assert torch.equal(a.q_rm, c.q_rm) and torch.equal(a.q_t, c.q_t) and torch.equal(a.scale, c.scale)


@pytest.mark.gpu
@pytest.mark.parametrize("ids", [np.arange(5, 7), torch.tensor([5, 6]), (5, np.int64(6)), range(5, 7), [5.0, "6"], {0: 5, 1: 6}])
def test_tensor_ids_of_any_kind_name_the_same_rounding_streams(ids):
    xs = [torch.randn(64, 96, device="cuda").to(torch.bfloat16) for _ in range(2)]
    ref = binding.fp4q_quantize2d_multi(xs, mode=binding.ROUND_STOCHASTIC, seed=7, tensor_ids=[5, 6])
    got = binding.fp4q_quantize2d_multi(xs, mode=np.int32(binding.ROUND_STOCHASTIC), seed=torch.tensor(7), tensor_ids=ids)
    for a, b in zip(ref, got):
        assert torch.equal(a.q_rm, b.q_rm) and torch.equal(a.q_t, b.q_t) and torch.equal(a.scale, b.scale)


@pytest.mark.gpu
def test_numbers_from_numpy_in_every_call():
    x, w = (torch.randn(256, 256, device="cuda").to(torch.bfloat16) for _ in range(2))
    n, i64 = np.int64(256), np.int64
    q = binding.fp4q_quantize2d(x, mode=i64(1), seed=i64(3), tensor_id=np.uint32(2), flags=np.uint32(0))
    same = binding.fp4q_quantize2d(x, mode=1, seed=3, tensor_id=2)
    assert torch.equal(q.q_rm, same.q_rm)
    qw = binding.fp4q_quantize2d(w)
    assert torch.equal(binding.fp4q_gemm_fwd(q, qw, dt=i64(1)), binding.fp4q_gemm_fwd(q, qw, dt=1))
    a, b = binding.fp4q_quantize1d(x, mode=i64(1), seed=i64(3), tensor_id=i64(2)), binding.fp4q_quantize1d(x, mode=1, seed=3, tensor_id=2)
    assert torch.equal(a[0], b[0])
    assert torch.equal(binding.fp4q_gemm_fwd_act1d(*a, n, qw, dt=i64(1)), binding.fp4q_gemm_fwd_act1d(*b, 256, qw, dt=1))
    xq, xs = binding.fp4q_mxfp8_quantize1d(x)
    assert torch.equal(binding.fp4q_mxfp8_gemm(xq, xs, xq, xs, n, n, n, dt=i64(0)), binding.fp4q_mxfp8_gemm(xq, xs, xq, xs, 256, 256, 256))
    f, g = (binding.fp4q_gemm_fwd_quantized(q, qw, mode=m, seed=s, tensor_id=t) for m, s, t in ((1, 5, 6), (i64(1), i64(5), i64(6))))
    assert torch.equal(f.q_rm, g.q_rm) and torch.equal(f.q_t, g.q_t) and torch.equal(f.scale, g.scale)
