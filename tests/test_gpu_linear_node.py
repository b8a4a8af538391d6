"""The layer's native autograd node against the Python function that does the same through the binding's calls."""
import threading

import pytest
import torch

from paper_2607_24953_b200 import autograd, binding

pytestmark = pytest.mark.gpu


def python_layer(x, w, seed, tensor_id, ws):
    return autograd._FP4LinearFn.apply(x, w, seed, tensor_id, ws)


def leaves(T, N, K, xd, wd, transposed=False):
    g = torch.Generator(device="cuda").manual_seed(T + N + K)
    x = torch.randn((K, T) if transposed else (T, K), generator=g, device="cuda").to(xd)
    w = torch.randn((K, N) if transposed else (N, K), generator=g, device="cuda").to(wd)
    return (x.t() if transposed else x), (w.t() if transposed else w), torch.randn(T, N, generator=g, device="cuda")


@pytest.mark.parametrize("T,N,K", [(1, 1, 1), (33, 100, 70), (128, 256, 256), (300, 1003, 777)])
@pytest.mark.parametrize("xd,wd", [(torch.bfloat16, torch.float32), (torch.float32, torch.bfloat16), (torch.float16, torch.float32)])
@pytest.mark.parametrize("needs", [(True, True), (True, False), (False, True)])
@pytest.mark.parametrize("transposed", [False, True])
def test_outputs_and_gradients_are_the_python_functions(T, N, K, xd, wd, needs, transposed):
    x, w, dy = leaves(T, N, K, xd, wd, transposed)
    ws = binding.alloc_workspace("cuda")
    got, nodes = [], []
    for layer in (autograd.fp4_linear, python_layer):
        a, b = x.detach().requires_grad_(needs[0]), w.detach().requires_grad_(needs[1])
        y = layer(a, b, 2 ** 63 + 5, 9, ws)
        assert y.dtype == torch.bfloat16 and y.is_contiguous() and y.requires_grad
        nodes.append(type(y.grad_fn).__name__)
        y.backward(dy.to(y.dtype))
        got.append((y.detach(), a.grad, b.grad))
    assert nodes[0] != "_FP4LinearFnBackward" and nodes[1] == "_FP4LinearFnBackward"   # two ways to the same result
    for u, v in zip(*got):
        assert (u is None) == (v is None)
        assert u is None or (u.dtype == v.dtype and u.shape == v.shape and torch.equal(u, v))


def test_leading_dimensions_no_grad_and_the_module():
    x, w, _ = leaves(24, 64, 96, torch.bfloat16, torch.float32)
    ws = binding.alloc_workspace("cuda")
    want = python_layer(x, w, 0, 0, ws)
    assert torch.equal(autograd.fp4_linear(x.view(2, 3, 4, 96), w, ws=ws), want.view(2, 3, 4, 64))
    with torch.no_grad():
        y = autograd.fp4_linear(x, w.requires_grad_(), ws=ws)
    assert not y.requires_grad and torch.equal(y, want)
    layer = autograd.FP4Linear(96, 64)
    layer(x).sum().backward()
    assert layer.weight.grad.shape == (64, 96) and torch.isfinite(layer.weight.grad).all()


def test_what_was_refused_stays_refused():
    x, w, dy = leaves(32, 64, 96, torch.bfloat16, torch.float32)
    ws = binding.alloc_workspace("cuda")
    y = autograd.fp4_linear(x.requires_grad_(), w, ws=ws)
    y.sum().backward(retain_graph=True)
    with pytest.raises((RuntimeError, AttributeError)):
        y.sum().backward()
    with pytest.raises(binding.Fp4qError):
        autograd.fp4_linear(x, w[:, :64].contiguous(), ws=ws)           # contractions differ
    with pytest.raises(binding.Fp4qError):
        autograd.fp4_linear(x, w, ws=ws[:4])                            # a workspace that is too small
    for bad in (lambda: autograd.fp4_linear(x.cpu(), w, ws=ws), lambda: autograd.fp4_linear(x, w.cpu(), ws=ws), lambda: autograd.fp4_linear(x, w[0], ws=ws)):
        with pytest.raises(ValueError):
            bad()
    with pytest.raises(TypeError):
        autograd.fp4_linear(x, w, seed=None, ws=ws)
    for layer in (autograd.fp4_linear, lambda a, b, ws: python_layer(a, b, 0, 0, ws)):   # no rows: forward, but no weight gradient
        y = layer(x[:0], w.detach().requires_grad_(), ws=ws)
        assert y.shape == (0, 64)
        with pytest.raises(binding.Fp4qError):
            y.sum().backward()
    with pytest.raises(Exception):
        torch.vmap(lambda a: autograd.fp4_linear(a, w, ws=ws))(x.detach().view(2, 16, 96))
    with pytest.raises(Exception):
        torch.func.grad(lambda a: autograd.fp4_linear(a, w, ws=ws).float().sum())(x.detach())
    with torch.autograd.forward_ad.dual_level(), pytest.raises(Exception):
        autograd.fp4_linear(torch.autograd.forward_ad.make_dual(x.detach(), x.detach()), w, ws=ws)


def test_transforms_tracers_and_modes_see_the_python_function():
    x, w, _ = leaves(32, 64, 96, torch.bfloat16, torch.float32)
    ws = binding.alloc_workspace("cuda")
    assert autograd._plain(x, w) and autograd._plain(x, torch.nn.Parameter(w))

    class Sub(torch.Tensor):
        pass

    assert not autograd._plain(x.as_subclass(Sub), w) and not autograd._plain(x, w.cpu())
    from torch.utils._python_dispatch import TorchDispatchMode

    class Mode(TorchDispatchMode):
        def __torch_dispatch__(self, func, types, args=(), kwargs=None):
            return func(*args, **(kwargs or {}))

    with Mode():
        assert not autograd._plain(x, w)
        y = autograd.fp4_linear(x, w, ws=ws)
    assert torch.equal(y, autograd.fp4_linear(x, w, ws=ws))
    seen = []
    torch.vmap(lambda a: seen.append(autograd._plain(a, w)) or a)(x.view(2, 16, 96))
    with torch.autograd.forward_ad.dual_level():
        seen.append(autograd._plain(x, w))
    assert seen == [False, False]


def test_hooks_streams_and_threads():
    x, w, dy = leaves(64, 128, 256, torch.bfloat16, torch.float32)
    ws = binding.alloc_workspace("cuda")
    a = x.detach().requires_grad_()
    calls = []
    with torch.autograd.graph.saved_tensors_hooks(lambda t: calls.append(t) or t, lambda t: t):
        y = autograd.fp4_linear(a, w, 3, 4, ws)
    y.register_hook(lambda g: g * 2)
    y.backward(dy.to(y.dtype))
    b = x.detach().requires_grad_()
    python_layer(b, w, 3, 4, ws).backward((2 * dy.to(y.dtype)))
    assert not calls and torch.equal(a.grad, b.grad)

    want = python_layer(x, w, 0, 0, ws)
    out, errors = {}, []

    def work(i):
        try:
            stream, own = torch.cuda.Stream(), binding.alloc_workspace("cuda")
            stream.wait_stream(torch.cuda.default_stream())
            with torch.cuda.stream(stream):
                for _ in range(20):
                    c = x.detach().requires_grad_()
                    y = autograd.fp4_linear(c, w, 3, 4, own)
                    assert type(y.grad_fn).__name__ != "_FP4LinearFnBackward"
                    y.backward((2 * dy.to(y.dtype)))
                out[i] = (y.detach().clone(), c.grad.clone())
            stream.synchronize()
        except Exception as exc:   # noqa: BLE001
            errors.append(exc)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not errors
    for y, gx in out.values():
        assert torch.equal(y, want) and torch.equal(gx, b.grad)


@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("lazy", ["negative bit", "zeros without memory"])
def test_fp32_operands_whose_memory_does_not_hold_their_values(which, lazy):
    x, w, _ = leaves(20, 48, 64, torch.float32, torch.float32)
    ops = [x, w]
    ops[which] = torch._neg_view(ops[which]) if lazy == "negative bit" else torch._efficientzerotensor(ops[which].shape, device="cuda")
    ws = binding.alloc_workspace("cuda")
    y = autograd.fp4_linear(*ops, 0, 0, ws)
    assert torch.equal(y, python_layer(*ops, 0, 0, ws))
    plain = [x, w]
    plain[which] = -plain[which] if lazy == "negative bit" else torch.zeros(plain[which].shape, device="cuda")
    assert torch.equal(y, autograd.fp4_linear(*plain, 0, 0, ws))


def both_layers(x, w, dy):
    """Outputs and gradients of the native node and of the Python function for the same operands."""
    ws, got, nodes = binding.alloc_workspace("cuda"), [], []
    for layer in (autograd.fp4_linear, python_layer):
        a, b = x.detach().requires_grad_(), w.detach().requires_grad_()
        y = layer(a, b, 5, 3, ws)
        nodes.append(type(y.grad_fn).__name__)
        y.backward(dy.to(y.dtype))
        got.append((y.detach(), a.grad, b.grad))
    assert nodes[0] != "_FP4LinearFnBackward" and nodes[1] == "_FP4LinearFnBackward"
    return got


@pytest.mark.parametrize("rows", [(1, 48), (20, 1), (1, 1)])   # one activation row, one output feature, both
@pytest.mark.parametrize("pitch", [64, 70, 72, 257])
@pytest.mark.parametrize("xd,wd", [(torch.float32, torch.float32), (torch.bfloat16, torch.float32), (torch.float32, torch.bfloat16)])
def test_single_rows_cut_from_wider_buffers(rows, pitch, xd, wd):
    T, N = rows
    x, w, dy = leaves(20, 48, pitch, xd, wd)
    x, w, dy = x[:T, :64], w[:N, :64], dy[:T, :N]
    x, w = (x if T == 1 else x.contiguous()), (w if N == 1 else w.contiguous())
    assert x.is_contiguous() and w.is_contiguous() and (x if T == 1 else w).stride(0) == pitch
    for u, v in zip(*both_layers(x, w, dy)):
        assert u.dtype == v.dtype and torch.equal(u, v)


def test_without_the_private_names_the_python_function_runs(monkeypatch):
    x, w, dy = leaves(20, 48, 64, torch.bfloat16, torch.float32)
    want = both_layers(x, w, dy)[1]
    monkeypatch.delattr(torch._C, "_len_torch_function_stack")
    monkeypatch.setattr(autograd, "_observed", autograd._find_observers())
    a, b = x.detach().requires_grad_(), w.detach().requires_grad_()
    y = autograd.fp4_linear(a, b, 5, 3, binding.alloc_workspace("cuda"))
    assert type(y.grad_fn).__name__ == "_FP4LinearFnBackward"
    monkeypatch.undo()
    y.backward(dy.to(y.dtype))
    for u, v in zip((y.detach(), a.grad, b.grad), want):
        assert torch.equal(u, v)
