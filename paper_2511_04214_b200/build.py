"""Build libbro.so in-tree with nvcc for sm_100a (cross-compiles without a GPU) and the binding's call module with g++."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
SO = os.path.join(HERE, "libbro.so")
SOURCES = [os.path.join(CSRC, "bro.cu")]
CALL_SO = os.path.join(HERE, "_call.so")
CALL_SOURCE = os.path.join(CSRC, "call.cpp")
HEADER = os.path.join(HERE, "..", "include", "bro.h")


def _deps():
    out = [HEADER]
    for name in os.listdir(CSRC):
        if name.endswith((".cu", ".cuh", ".h")):
            out.append(os.path.join(CSRC, name))
    return out


def nvcc_command(verbose: bool = False):
    cmd = ["nvcc", "-std=c++17", "-O3", "-lineinfo",
           "-gencode", "arch=compute_100a,code=sm_100a",
           "-Xcompiler", "-fPIC", "-shared", "--fmad=false",
           "-o", SO] + SOURCES
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    return cmd


def call_tag() -> str:
    """What the call module is good for: it reads torch's tensors in place, so only the torch, the C++ ABI and the Python that it was
    compiled against may load it."""
    import torch
    return f"call module for torch {torch.__version__}, C++11 ABI {int(torch._C._GLIBCXX_USE_CXX11_ABI)}, {sysconfig.get_config_var('SOABI')}"


def call_command():
    import torch
    from torch.utils import cpp_extension
    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    include = cpp_extension.include_paths() + [sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    return (["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-fvisibility=hidden", "-w",
             f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DBRO_CALL_TAG="{call_tag()}"']
            + [f"-I{p}" for p in include] + ["-o", CALL_SO, CALL_SOURCE, "-L" + os.path.join(root, "lib")]
            + ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"])


def _stale(so, deps):
    return not os.path.exists(so) or os.path.getmtime(so) < max(os.path.getmtime(p) for p in deps)


def _call_stale():
    if _stale(CALL_SO, [HEADER, CALL_SOURCE]):
        return True
    with open(CALL_SO, "rb") as f:
        return call_tag().encode() + b"\0" not in f.read()


def build(force: bool = False, verbose: bool = False) -> str:
    call = None
    if force or _call_stale():
        call = subprocess.Popen(call_command())
    try:
        if force or _stale(SO, _deps()):
            subprocess.run(nvcc_command(verbose), check=True)
    finally:
        if call is not None and call.wait() != 0:
            raise subprocess.CalledProcessError(call.returncode, call.args)
    return SO


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(SO)
