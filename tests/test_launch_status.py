"""What a failed launch leaves behind: the quantizers' entry points, linked against a stand-in for the CUDA runtime."""
import ctypes
import os
import subprocess

import pytest

from paper_2607_24953_b200 import binding, build

HERE = os.path.dirname(os.path.abspath(__file__))
FP4Q_ERR_CUDA = 6
P = ctypes.c_void_p(1 << 20)   # an aligned address that nothing on the host reads


@pytest.fixture(scope="module")
def entries(tmp_path_factory):
    out = tmp_path_factory.mktemp("launch")
    objs, procs = [], []
    for name in ("quantize1d", "quantize2d", "mxfp8_quantize"):
        src, obj = os.path.join(build.CSRC, name + ".cu"), str(out / (name + ".o"))
        objs.append(obj)
        procs.append(subprocess.Popen(["nvcc"] + build.NVCC_FLAGS + ["-c", src, "-o", obj], stdout=subprocess.DEVNULL, stderr=subprocess.DEVNULL))
    assert all(p.wait() == 0 for p in procs)
    so = str(out / "entries.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-w", "-Wl,-Bsymbolic", "-o", so, os.path.join(HERE, "helpers", "fake_cudart.c")] + objs + ["-lstdc++"],
                   check=True)
    L = ctypes.CDLL(so)
    real = binding.lib()
    for name in ("fp4q_quantize2d", "fp4q_quantize2d_multi", "fp4q_quantize1d", "fp4q_quantize1d_t", "fp4q_mxfp8_quantize1d", "fp4q_mxfp8_quantize1d_t"):
        getattr(L, name).argtypes = getattr(real, name).argtypes
    return L


def _calls(L):
    rows, cols = 128, 256
    t = binding._CTensor(rows, cols, P.value, cols // 2, P.value, rows // 2, P.value, cols // 32)
    jobs = (binding._CQuantJob * 2)(*[binding._CQuantJob(P.value, rows, cols, cols, ctypes.pointer(t), j, 0) for j in range(2)])
    return {"quantize2d": lambda: L.fp4q_quantize2d(P, rows, cols, cols, ctypes.byref(t), 1, 0, 0, 0, None),
            "quantize2d_multi": lambda: L.fp4q_quantize2d_multi(jobs, 2, 0, 0, None),
            "quantize1d": lambda: L.fp4q_quantize1d(P, rows, cols, cols, P, cols // 2, P, cols // 32, 0, 0, 0, None),
            "quantize1d stochastic": lambda: L.fp4q_quantize1d(P, rows, cols, cols, P, cols // 2, P, cols // 32, 1, 0, 0, None),
            "quantize1d_t": lambda: L.fp4q_quantize1d_t(P, rows, cols, cols, P, rows // 2, P, rows // 32, None),
            "quantize1d_t ragged": lambda: L.fp4q_quantize1d_t(P, rows - 1, cols, cols, P, rows // 2, P, rows // 32, None),
            "mxfp8_quantize1d": lambda: L.fp4q_mxfp8_quantize1d(P, rows, cols, cols, P, cols, P, cols // 32, None),
            "mxfp8_quantize1d_t": lambda: L.fp4q_mxfp8_quantize1d_t(P, rows, cols, cols, P, rows, P, rows // 32, None),
            "mxfp8_quantize1d_t ragged": lambda: L.fp4q_mxfp8_quantize1d_t(P, rows - 1, cols, cols, P, rows, P, rows // 32, None)}


def test_a_launch_reports_its_own_error_only(entries):
    for name, call in _calls(entries).items():
        entries.fake_set(0, 0)
        assert call() == 0 and entries.fake_last_error() == 0, name
        entries.fake_set(0, 101)                 # somebody else's leftover
        assert call() == 0 and entries.fake_last_error() == 101, name
        entries.fake_set(98, 0)                  # this launch fails
        assert call() == FP4Q_ERR_CUDA and entries.fake_last_error() == 0, name
