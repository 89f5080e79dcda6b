"""Builds libmoc_b200.so (nvcc, sm_100a only) and _moc_torch.so (g++: the torch side of the binding)
next to this file.  ``python -m paper_2304_14463_b200.build``"""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmoc_b200.so")
SOURCES = ["moc_api.cu", "moc_search.cu", "moc_intervals.cu", "moc_edits.cu", "moc_eval_general.cu", "moc_eval_pair.cu", "moc_eval_lane.cu",
           "moc_eval_quad.cu", "moc_eval_quad_warp.cu", "moc_eval_live.cu", "moc_check_plain.cu", "moc_check_general.cu", "moc_check_staged.cu", "moc_search_score.cu", "moc_search_walk.cu", "moc_search_walk_floor.cu"]
HEADERS = ["moc_kernels.cuh", "moc_pair_kernel.cuh", "moc_lane_kernel.cuh", "moc_quad_kernel.cuh", "moc_live_kernel.cuh", "moc_host.cuh", "moc_search_kernels.cuh", "moc_search_score_kernel.cuh", "moc_search_walk_kernel.cuh", "moc_edit_pass.cuh", "moc_edit_lanes_kernel.cuh", "moc_interval_kernels.cuh", "moc_interval_plain_kernel.cuh", "moc_edit_kernels.cuh", "moc_cache_host.cuh", os.path.join("..", "..", "include", "moc.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-shared", "--use_fast_math"]


TORCH_LIB = os.path.join(HERE, "_moc_torch.so")
TORCH_KEY = TORCH_LIB + ".key"      # torch and Python that _moc_torch.so was built for
TORCH_SOURCES = ["moc_torch.cpp", os.path.join("..", "..", "include", "moc.h")]


def _stale(lib, files):
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = [os.path.join(CSRC, f) for f in files] + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def torch_key() -> str:
    import torch
    return f"torch {torch.__version__} cxx11abi {int(torch._C._GLIBCXX_USE_CXX11_ABI)} {sys.implementation.cache_tag}"


def torch_lib_fits() -> bool:
    """Whether _moc_torch.so was built for this torch (its C++ interface is not stable) and Python."""
    try:
        with open(TORCH_KEY) as f:
            return os.path.exists(TORCH_LIB) and f.read() == torch_key()
    except OSError:
        return False


def build_torch(force: bool = False) -> str:
    if not force and torch_lib_fits() and not _stale(TORCH_LIB, TORCH_SOURCES):
        return TORCH_LIB
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    lib_dirs = [os.path.join(os.path.dirname(torch.__file__), "lib")]
    tmp = TORCH_LIB + f".{os.getpid()}.tmp"
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    cmd += [f"-I{d}" for d in cpp_extension.include_paths("cuda") + [sysconfig.get_paths()["include"]]]
    cmd += ["-o", tmp, os.path.join(CSRC, "moc_torch.cpp")]
    cmd += [f for d in lib_dirs for f in (f"-L{d}", f"-Wl,-rpath,{d}")]
    cmd += ["-lc10", "-lc10_cuda", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, TORCH_LIB)
    with open(TORCH_KEY, "w") as f:
        f.write(torch_key())
    return TORCH_LIB


def build(force: bool = False, verbose: bool = False) -> str:
    build_torch(force)
    if not force and not _stale(LIB, SOURCES + HEADERS):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
          ["-t", "8", "-o", tmp] + [os.path.join(CSRC, f) for f in SOURCES]
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
