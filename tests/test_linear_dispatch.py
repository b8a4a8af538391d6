"""The layer's choice between its native node and its Python function, as far as it needs no GPU."""
import pytest
import torch
from torch.autograd import forward_ad

from paper_2607_24953_b200 import autograd


def test_what_looks_into_python_functions_is_seen():
    assert autograd._observed() is False
    seen = []
    torch.vmap(lambda a: seen.append(autograd._observed()) or a)(torch.zeros(2, 3))
    with forward_ad.dual_level():
        seen.append(autograd._observed())
    with torch.device("cpu"):   # a function mode
        seen.append(autograd._observed())
    torch.jit.trace(lambda a: (seen.append(autograd._observed()), a + 1)[1], (torch.zeros(2),), check_trace=False)
    assert seen == [True] * 4 and autograd._observed() is False


@pytest.mark.parametrize("where,name", [(torch._C, "_len_torch_function_stack"), (torch._C, "_len_torch_dispatch_stack"), (torch._C, "_get_tracing_state"),
                                        (torch._C._functorch, "peek_interpreter_stack"), (forward_ad, "_current_level"), (torch.compiler, "is_compiling")])
def test_a_torch_without_one_of_the_names_takes_the_python_function(monkeypatch, where, name):
    monkeypatch.delattr(where, name)
    found = autograd._find_observers()
    monkeypatch.undo()
    assert found is None
    monkeypatch.setattr(autograd, "_observed", found)

    class OnGpu:   # what _plain asks of a tensor
        is_cuda, device = True, "cuda:0"
        def dim(self): return 2

    monkeypatch.setattr(autograd, "_TENSORS", (OnGpu,))
    assert autograd._plain(OnGpu(), OnGpu()) is False
    monkeypatch.undo()
    monkeypatch.setattr(autograd, "_TENSORS", (OnGpu,))
    assert autograd._plain(OnGpu(), OnGpu()) is True
