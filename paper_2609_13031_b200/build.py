"""Build libfp8attn.so (CUDA, sm_100a only) in-tree with nvcc, and the native half of its Python binding with g++."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
LIB = os.path.join(_HERE, "libfp8attn.so")
SOURCES = ["api.cu", "quantize.cu", "attention.cu", "perturb.cu", "host_step.cu", "key_order.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _stale(target: str, deps: list[str]) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build_cuda(force: bool = False, verbose: bool = False) -> str:
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    headers.append(os.path.join(INCLUDE, "fp8attn.h"))
    objs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(CSRC, src.replace(".cu", ".o"))
        if force or _stale(o, [s] + headers):
            cmd = [_nvcc(), *NVCC_FLAGS, "-I", INCLUDE, "-I", CSRC, "-c", s, "-o", o]
            if verbose:
                cmd.insert(1, "-Xptxas=-v")
            subprocess.run(cmd, check=True)
        objs.append(o)
    if force or _stale(LIB, objs):
        tmp = LIB + f".tmp{os.getpid()}"
        subprocess.run([_nvcc(), "-shared", "-o", tmp, *objs, "-cudart", "static"], check=True)
        os.replace(tmp, LIB)
    return LIB


def binding_path() -> str:
    """Where the native half of the binding stands for this interpreter and this torch, whose C++ interface it is
    compiled against: another one finds no file there instead of one that does not fit."""
    import torch
    return os.path.join(_HERE, f"_binding.{sys.implementation.cache_tag}.torch-{torch.__version__}.so")


def build_binding(force: bool = False) -> str:
    """csrc/binding.cpp against this torch: a CPython module beside the library."""
    import torch
    from torch.utils import cpp_extension
    src, target = os.path.join(CSRC, "binding.cpp"), binding_path()
    if force or _stale(target, [src, os.path.join(INCLUDE, "fp8attn.h")]):
        system = cpp_extension.include_paths("cuda") + [sysconfig.get_paths()["include"]]
        tmp = target + f".tmp{os.getpid()}"
        subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
                        f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}", "-I", INCLUDE,
                        *(a for d in system for a in ("-isystem", d)), src, "-o", tmp,
                        "-L" + os.path.join(os.path.dirname(torch.__file__), "lib"),
                        "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"], check=True)
        os.replace(tmp, target)
    return target


if __name__ == "__main__":
    print(build_cuda(force="--force" in sys.argv, verbose="-v" in sys.argv))
    print(build_binding(force="--force" in sys.argv))
