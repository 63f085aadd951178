"""Builds the CUDA library in-tree: nvcc -> paper_2405_03917_b200/libcq.so (sm_100a only), and the native side of the
Python binding: g++ -> paper_2405_03917_b200/_cq_native.so."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcq.so")
NATIVE = os.path.join(HERE, "_cq_native.so")
SOURCES = ["cq_api.cu", "cq_generic.cu", "cq_encode.cu", "cq_encode_tc.cu", "cq_encode_grid.cu", "cq_decode.cu", "cq_decode_pair.cu", "cq_decode_rope.cu", "cq_decode_tables.cu", "cq_prefill.cu", "cq_learn.cu", "cq_learn_assign.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--cudart", "shared", "-Xlinker", "-rpath=/usr/local/cuda/lib64"]


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(NATIVE):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(NATIVE))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(HERE, "..", "include", "cq.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    flags = list(NVCC_FLAGS)
    if verbose:
        flags += ["-Xptxas", "-v"]
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc, *flags, "-shared", "-o", tmp, *[os.path.join(CSRC, s) for s in SOURCES]]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    build_native()
    return LIB


def build_native() -> str:
    """The CPython extension of the hot calls: torch headers, linked against libcq.so beside it."""
    import sysconfig

    import torch
    from torch.utils import cpp_extension
    tmp = NATIVE + ".tmp.%d" % os.getpid()
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           *["-I" + p for p in cpp_extension.include_paths()], "-I" + sysconfig.get_paths()["include"],
           "-I" + os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"),
           os.path.join(CSRC, "cq_binding.cpp"), "-o", tmp, "-L" + HERE, "-l:libcq.so", "-Wl,-rpath,$ORIGIN",
           *["-L" + p for p in cpp_extension.library_paths()], "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    subprocess.check_call(cmd)
    os.replace(tmp, NATIVE)
    return NATIVE


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
