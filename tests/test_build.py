"""When the marshalling module counts as built, and what is said when it does not load."""
import os
import sys

import pytest
import torch

from paper_2607_24953_b200 import binding, build


@pytest.fixture
def built(tmp_path, monkeypatch):
    for name, text in (("HOST", "so"), ("HOST_STAMP", "")):
        path = tmp_path / name
        path.write_text(text)
        monkeypatch.setattr(build, name, str(path))
    (tmp_path / "HOST_STAMP").write_text(build.host_stamp())
    return tmp_path


def test_a_module_of_this_python_and_torch_is_kept(built):
    assert not build.host_stale()


@pytest.mark.parametrize("change", ["torch", "python", "flags", "stamp", "module"])
def test_a_module_of_another_torch_python_or_command_is_rebuilt(built, monkeypatch, change):
    if change == "torch":
        monkeypatch.setattr(torch, "__version__", "0.0.0")
    elif change == "python":
        monkeypatch.setattr(build.sysconfig, "get_config_var", lambda name: "cpython-0")
    elif change == "flags":
        command = build.host_command
        monkeypatch.setattr(build, "host_command", lambda out: command(out) + ["-O0"])
    else:
        (built / {"stamp": "HOST_STAMP", "module": "HOST"}[change]).unlink()
    assert build.host_stale()


def test_a_module_that_does_not_load_is_told_from_one_that_is_missing(tmp_path, monkeypatch):
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(binding, "_HERE", str(tmp_path))
    with pytest.raises(ImportError, match="not built"):
        binding._host()
    (tmp_path / "_host.so").write_bytes(b"not a shared object")
    monkeypatch.setitem(sys.modules, "paper_2607_24953_b200._host", None)      # what an import that fails looks like
    monkeypatch.delattr(sys.modules["paper_2607_24953_b200"], "_host", raising=False)
    with pytest.raises(ImportError, match="does not load"):
        binding._host()
    assert os.path.exists(build.HOST)
