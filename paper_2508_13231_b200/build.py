"""Builds libkvp.so (sm_100a only) in-tree with nvcc, and _kvp_torch.so, the native side of the Python binding, with g++.
Usable as `python -m paper_2508_13231_b200.build`."""
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libkvp.so")
BINDING = os.path.join(HERE, "_kvp_torch.so")
SOURCES = ["kvp_api.cu", "kvp_cost.cu", "kvp_layout.cu", "kvp_anneal.cu", "kvp_trace.cu", "kvp_policy.cu", "kvp_table.cpp"]
HEADERS = ["kvp_common.cuh", "kvp_chain.cuh", "kvp_narrow.cuh"]


def _nvcc():
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _fresh(target, deps):
    return os.path.exists(target) and all(os.path.getmtime(target) >= os.path.getmtime(d) for d in deps)


def build_binding(force=False):
    src = os.path.join(CSRC, "kvp_torch.cpp")
    if not force and _fresh(BINDING, [src, os.path.join(HERE, "..", "include", "kvp.h")]):
        return BINDING
    import sysconfig

    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    subprocess.check_call(
        [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-w", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
         f"-I{sysconfig.get_path('include')}", f"-I{root}/include", f"-I{root}/include/torch/csrc/api/include", f"-I{cuda}/include",
         src, "-o", BINDING, f"-L{HERE}", "-l:libkvp.so", "-Wl,-rpath,$ORIGIN", f"-L{root}/lib", "-ltorch_python", "-ltorch_cuda",
         "-ltorch_cpu", "-lc10_cuda", "-lc10"])
    return BINDING


def build_library(force=False, verbose=False):
    srcs = [os.path.join(CSRC, s) for s in SOURCES]
    deps = srcs + [os.path.join(CSRC, h) for h in HEADERS] + [os.path.join(HERE, "..", "include", "kvp.h")]
    if force or not _fresh(LIB, deps):
        cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
               "-shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-ffp-contract=off", "-Xlinker", "-soname=libkvp.so", "-o", LIB] + srcs
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        subprocess.check_call(cmd)
    build_binding(force)
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
