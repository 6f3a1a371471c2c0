"""Builds libuniql.so (the C-ABI CUDA library, nvcc for sm_100a) and _calls.so (its Python entry points, g++) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libuniql.so")
CALLS = os.path.join(HERE, "_calls.so")
SOURCES = ["api.cu", "util_kernels.cu", "generic.cu", "decode.cu", "gemv.cu", "prefill.cu", "single.cu", "batch.cu", "noalloc.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
              "-Xcompiler", "-fPIC", "--use_fast_math=false"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _stale() -> bool:
    if not (os.path.exists(LIB) and os.path.exists(CALLS)):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(CALLS))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(HERE, "..", "include", "uniql.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _newest(src: str) -> float:
    """Time of the last change to a source file or to a header that it may include."""
    heads = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    return max(os.path.getmtime(f) for f in heads + [os.path.join(CSRC, src), os.path.join(HERE, "..", "include", "uniql.h")])


def _calls_cmd(out: str) -> list:
    """g++ command for the Python entry points; libtorch and libuniql.so are found where the process has loaded them."""
    import torch
    from torch.utils import cpp_extension
    inc = [d for d in cpp_extension.include_paths() if os.path.isdir(d)]
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    inc += [os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    return (["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-w", "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch.compiled_with_cxx11_abi()]
            + sum((["-isystem", d] for d in inc), []) + [os.path.join(CSRC, "pybind.cpp"), "-o", out]
            + ["-L" + d for d in cpp_extension.library_paths()]
            + ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-L" + HERE, "-l:libuniql.so", "-Wl,-rpath,$ORIGIN"])


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    objs = []
    bdir = os.path.join(HERE, "_build")
    os.makedirs(bdir, exist_ok=True)
    flags = [f for f in NVCC_FLAGS if not f.startswith("--use_fast_math")]
    if verbose:
        flags += ["-Xptxas", "-v"]
    procs = []
    for src in SOURCES:
        obj = os.path.join(bdir, src.replace(".cu", ".o"))
        objs.append(obj)
        if not force and not verbose and os.path.exists(obj) and os.path.getmtime(obj) > _newest(src):
            continue
        cmd = [_nvcc()] + flags + ["-c", os.path.join(CSRC, src), "-o", obj]
        procs.append((cmd, subprocess.Popen(cmd)))
    for cmd, pr in procs:
        if pr.wait() != 0:
            raise RuntimeError("nvcc failed: " + " ".join(cmd))
    tmp = LIB + ".%d.tmp" % os.getpid()
    subprocess.check_call([_nvcc(), "-shared", "-Xlinker", "-soname,libuniql.so", "-o", tmp] + objs + ["-lcudart"])
    os.replace(tmp, LIB)
    if force or not os.path.exists(CALLS) or os.path.getmtime(CALLS) < _newest("pybind.cpp"):
        tmp = CALLS + ".%d.tmp" % os.getpid()
        subprocess.check_call(_calls_cmd(tmp))
        os.replace(tmp, CALLS)
    else:
        os.utime(CALLS)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
