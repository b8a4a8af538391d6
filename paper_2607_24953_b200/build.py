"""Builds libfp4q.so (the C-ABI CUDA library, nvcc, sm_100a) and _host.so (the binding's native marshalling, g++) in-tree."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libfp4q.so")
HOST_SRC = os.path.join(CSRC, "host", "marshal.cpp")
HOST = os.path.join(HERE, "_host.so")
HOST_STAMP = os.path.join(HERE, "build", "_host.stamp")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I" + INCLUDE, "-I" + CSRC]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def host_command(out: str):
    """g++ of the marshalling module, against the Python that runs and the headers and libraries of the torch it imports."""
    import torch
    nvcc = shutil.which("nvcc")
    cuda = os.environ.get("CUDA_HOME") or (os.path.dirname(os.path.dirname(os.path.realpath(nvcc))) if nvcc else "/usr/local/cuda")
    root = os.path.dirname(torch.__file__)
    inc = [INCLUDE, sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    sysinc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include")]
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch.compiled_with_cxx11_abi())]
    cmd += ["-I" + d for d in inc] + [a for d in sysinc for a in ("-isystem", d)]
    return cmd + ["-o", out, HOST_SRC, "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def host_stamp() -> str:
    """What a built _host.so is good for: this Python, this torch, this way of building it (wherever the tree lies)."""
    import torch
    command = " ".join(host_command(HOST)).replace(os.path.dirname(HERE), ".")
    return "\n".join([sysconfig.get_config_var("SOABI") or sys.version, torch.__version__, str(torch.version.cuda), command])


def host_stale() -> bool:
    if not os.path.exists(HOST) or not os.path.exists(HOST_STAMP):
        return True
    t = os.path.getmtime(HOST)
    if any(os.path.getmtime(d) > t for d in [HOST_SRC] + glob.glob(os.path.join(INCLUDE, "*.h"))):
        return True
    with open(HOST_STAMP) as f:
        return f.read() != host_stamp()


def start_host_build():
    tmp = HOST + ".%d.tmp" % os.getpid()
    return tmp, subprocess.Popen(host_command(tmp), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)


def finish_host_build(tmp, pr):
    out, _ = pr.communicate()
    if pr.returncode != 0:
        sys.stderr.write(out)
        raise RuntimeError("g++ failed on %s" % HOST_SRC)
    if os.path.exists(HOST_STAMP):
        os.remove(HOST_STAMP)
    os.replace(tmp, HOST)
    with open(HOST_STAMP, "w") as f:
        f.write(host_stamp())


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every csrc/*.cu and link libfp4q.so, and the marshalling module. Returns the library path."""
    os.makedirs(os.path.join(HERE, "build"), exist_ok=True)
    host = start_host_build() if force or host_stale() else None
    try:
        return build_library(force, verbose)
    finally:
        if host:
            finish_host_build(*host)


def build_library(force: bool = False, verbose: bool = False) -> str:
    if not force and not stale():
        return LIB
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    objs = []
    procs = []
    for src in sources():
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        cmd = ["nvcc"] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    for src, pr in procs:
        out, _ = pr.communicate()
        if verbose or pr.returncode != 0:
            sys.stderr.write(out)
        if pr.returncode != 0:
            raise RuntimeError("nvcc failed on %s" % src)
    tmp = LIB + ".%d.tmp" % os.getpid()
    subprocess.run(["nvcc", "-shared", "-o", tmp] + objs + ["-ldl"], check=True)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
