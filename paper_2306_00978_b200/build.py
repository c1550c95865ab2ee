"""Builds the CUDA library in-tree with nvcc for sm_100a (no JIT cache), and the binding's native
call paths (csrc/native_calls.cpp, a CPython module on torch's C++ interface) with g++.

    python -m paper_2306_00978_b200.build            # build if sources are newer
    python -m paper_2306_00978_b200.build --force
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB_NAME = "libawq_b200.so"
LIB_PATH = os.path.join(HERE, LIB_NAME)
NATIVE_PATH = os.path.join(HERE, "_native.so")
SOURCES = ("api.cu", "quantize_pack.cu", "gemv.cu", "gemv_mid.cu", "gemm_tcgen05.cu", "gemm_tcgen05_pair.cu", "gemm_stream.cu", "search.cu")
NVCC_FLAGS = (
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "--std=c++17",
    "-Xcompiler", "-fPIC",
)


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(NATIVE_PATH):
        return True
    t = min(os.path.getmtime(LIB_PATH), os.path.getmtime(NATIVE_PATH))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".o")]
    deps.append(os.path.join(os.path.dirname(HERE), "include", "awq_b200.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def _native_command() -> list:
    import torch
    from torch.utils import cpp_extension
    includes = [*cpp_extension.include_paths(), os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include"),
                sysconfig.get_paths()["include"]]
    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-o", NATIVE_PATH,
            os.path.join(CSRC, "native_calls.cpp"), f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
            *[f"-isystem{i}" for i in includes], f"-L{libs}", "-ltorch_python", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-lc10",
            "-lc10_cuda"]


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every kernel for sm_100a into one shared library; returns its path."""
    out = LIB_PATH
    if not force and not _stale():
        return LIB_PATH
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        cmd = [_nvcc(), *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    procs.append(("native_calls.cpp", subprocess.Popen(_native_command(), stdout=subprocess.PIPE,
                                                       stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        log, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(log)
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("compilation failed")
    link = [_nvcc(), "-shared", "-o", out, *objs, "-lcudart", "-Xcompiler", "-fPIC"]
    subprocess.run(link, check=True)
    return out


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
