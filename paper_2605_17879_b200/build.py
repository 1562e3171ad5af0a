"""Builds the CUDA library in-tree with nvcc for sm_100a (B200)."""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libguard_b200.so")
NATIVE = os.path.join(HERE, "_guard_native.so")   # the Python binding's marshalling (csrc/binding.cpp)
SOURCES = ["guard_api.cu", "xrank.cu", "xrank_bracket.cu", "xrank_cluster.cu", "xrank_split.cu", "xrank_count.cu", "window.cu", "window_bins.cu", "score.cu", "topk.cu", "eval_tail.cu", "sweep.cu", "triage.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--fmad=false",            # every decision is defined on unfused float32 operations
    "-Xcompiler", "-fPIC",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(NATIVE):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(NATIVE))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(HERE, "..", "include", "guard_b200.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _build_native() -> None:
    """The marshalling module: linked to the library next to it and to the libraries torch has loaded."""
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    tmp = NATIVE + ".%d.tmp" % os.getpid()
    tlib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-w",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), "-I" + sysconfig.get_paths()["include"],
           *["-I" + d for d in cpp_extension.include_paths()], "-I" + os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include"),
           os.path.join(CSRC, "binding.cpp"), "-o", tmp, "-L" + HERE, "-L" + tlib, "-l:libguard_b200.so", "-lc10", "-lc10_cuda",
           "-ltorch_cpu", "-ltorch_python", "-Wl,-rpath,$ORIGIN"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("g++ failed on binding.cpp")
    os.replace(tmp, NATIVE)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu into libguard_b200.so next to this file, and the binding's module; returns the library's path."""
    if not force and not _stale():
        return LIB
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    nvcc = _nvcc()
    extra = ["-Xptxas", "-v"] if verbose else []

    def compile_one(src: str) -> str:
        obj = os.path.join(objdir, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, *extra, "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed on " + src)
        return obj

    with ThreadPoolExecutor(max_workers=min(8, len(SOURCES))) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + ".%d.tmp" % os.getpid()
    subprocess.check_call([nvcc, "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a"])
    os.replace(tmp, LIB)
    _build_native()
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
