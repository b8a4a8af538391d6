"""A process's and a thread's first product: the host code of the products' entry points, linked against a stand-in for the CUDA runtime."""
import ctypes
import os
import subprocess
import threading

import pytest

from paper_2607_24953_b200 import binding, build

HERE = os.path.dirname(os.path.abspath(__file__))
P = 1 << 20   # an aligned address that nothing on the host reads


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    out = tmp_path_factory.mktemp("first")
    so, objs = str(out / "gemm.so"), [str(out / "gemm.o"), str(out / "api.o")]
    flags = [f.replace("code=sm_100a", "code=compute_100a") for f in build.NVCC_FLAGS]   # the device code is not run
    for obj, name in zip(objs, ("gemm_blockscaled.cu", "api.cu")):
        subprocess.run(["nvcc"] + flags + ["-c", os.path.join(build.CSRC, name), "-o", obj], check=True, stdout=subprocess.DEVNULL, stderr=subprocess.DEVNULL)
    subprocess.run(["gcc", "-shared", "-fPIC", "-w", "-Wl,-Bsymbolic", "-o", so, os.path.join(HERE, "helpers", "fake_cudart_gemm.c")] + objs + ["-lstdc++"], check=True)
    return so


def product(L, bind):
    """One forward product of 300 x 512 x 256; the status."""
    f = L.fp4q_gemm_fwd
    f.argtypes = binding.lib().fp4q_gemm_fwd.argtypes
    x, w = (binding._CTensor(rows, 256, P, 128, P, 512, P, 8) for rows in (512, 300))
    if bind:
        L.fake_bind()
    return f(ctypes.byref(x), ctypes.byref(w), P, 304, 0, None, P, 1 << 20, None)


def in_threads(n, call):
    status, gate = [None] * n, threading.Barrier(n)
    def work(i):
        gate.wait()
        status[i] = call()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(n)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return status


def test_first_products_of_several_threads(library):
    # all come while the first of them looks for the driver's entry point
    L = ctypes.CDLL(library)
    assert in_threads(8, lambda: product(L, True)) == [0] * 8


def test_a_threads_first_call_is_a_product(library):
    # nothing has bound the thread to a device: the encoder refuses it, the product binds it and goes on
    L = ctypes.CDLL(library)
    assert in_threads(2, lambda: (product(L, False), L.fake_bound())) == [(0, 1)] * 2


@pytest.mark.gpu
def test_a_threads_first_call_is_a_product_on_the_device():
    import torch
    from paper_2607_24953_b200 import workloads
    qx, qw = (binding.fp4q_quantize2d(workloads.activations_student_t(rows, 256, rows, "cuda")) for rows in (512, 300))
    ws, out = binding.alloc_workspace("cuda"), torch.zeros(2, 512, 304, dtype=torch.bfloat16, device="cuda")[:, :, :300]
    binding.fp4q_gemm_fwd(qx, qw, out=out[0], ws=ws)
    torch.cuda.synchronize()
    in_threads(1, lambda: binding.fp4q_gemm_fwd(qx, qw, out=out[1], ws=ws))
    torch.cuda.synchronize()
    assert out[0].any() and torch.equal(out[0], out[1])
