"""Build the sr_gate CUDA library in-tree with nvcc for sm_100a, and the Python extension around it.

    python -m paper_2605_05802_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsr_gate.so")
NATIVE = os.path.join(HERE, "_native.so")
BINDING = os.path.join(CSRC, "torch_binding.cpp")
SOURCES = ["api.cu", "gate_single.cu", "gate_multi.cu", "incremental.cu", "advantage.cu", "probe.cu",
           "gate_noalloc.cu", "signals.cu", "gate_packed.cu", "compact.cu"]


def _stale(target: str, sources) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    deps = list(sources) + [os.path.join(ROOT, "include", f) for f in os.listdir(os.path.join(ROOT, "include"))]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    sources = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))]
    if force or _stale(LIB, sources):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
               "-Xcompiler", "-fPIC", "-shared", "-cudart", "static", "--threads", "0",
               "-I", os.path.join(ROOT, "include"), "-I", CSRC]
        if verbose:
            cmd += ["-Xptxas", "-v"]
        cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", tmp]
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    if force or _stale(NATIVE, [BINDING]):
        build_native()
    return LIB


def build_native() -> str:
    """The Python extension around the library (host code only)."""
    import torch
    from torch.utils import cpp_extension
    tmp = NATIVE + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
           "-I", os.path.join(ROOT, "include"), "-isystem", sysconfig.get_paths()["include"]]
    for d in cpp_extension.include_paths("cuda"):
        cmd += ["-isystem", d]
    cmd += [BINDING, "-o", tmp, "-L", HERE, "-lsr_gate", "-Wl,-rpath,$ORIGIN"]
    for d in cpp_extension.library_paths():
        cmd += ["-L", d]
    cmd += ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    subprocess.check_call(cmd)
    os.replace(tmp, NATIVE)
    return NATIVE


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
