"""Builds libgsa.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _native.*.so, through which the binding takes
torch tensors into its decode step.  The latter is compiled against this interpreter and this torch, whose versions its name
has; nothing but the speed of the decode call depends on it, so where it cannot be built the build says so and goes on.

    python -m paper_2409_07146_b200.build [--force] [--verbose]

nvcc cross-compiles, so this works on a machine without a GPU.  The shared
object is written next to this file; it is git-ignored but travels with the
source tree.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

from .binding import native_path

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libgsa.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
    "--expt-relaxed-constexpr",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _build_native() -> None:
    import torch
    from torch.utils import cpp_extension
    path = native_path()
    tmp = path + ".tmp.%d" % os.getpid()
    cuda = os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include")
    include = [os.path.join(ROOT, "include"), sysconfig.get_paths()["include"], cuda, *cpp_extension.include_paths()]
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
                           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), *["-I" + d for d in include],
                           os.path.join(CSRC, "binding_native.cpp"), "-o", tmp, "-L" + lib, "-ltorch_python", "-ltorch_cpu", "-lc10_cuda",
                           "-lc10"])
    os.replace(tmp, path)
    for old in glob.glob(os.path.join(HERE, "_native*.so")):
        if old != path:
            os.remove(old)


def _stale(path: str, deps) -> bool:
    headers = glob.glob(os.path.join(ROOT, "include", "*.h")) + [os.path.abspath(__file__)]
    return not os.path.exists(path) or any(os.path.getmtime(d) > os.path.getmtime(path) for d in [*deps, *headers])


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh"))):
        _build_library(verbose)
    if force or _stale(native_path(), [os.path.join(CSRC, "binding_native.cpp")]):
        try:
            _build_native()
        except Exception as e:
            print(f"not built: {native_path()} ({e}); decode calls go through Python, a few microseconds slower", file=sys.stderr)
    return LIB


def _build_library(verbose: bool) -> None:
    objs = []
    procs = []
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    flags = [f for f in NVCC_FLAGS if f != "--shared"]
    for src in sources():
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        cmd = [NVCC, *flags, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd)))
        objs.append(obj)
    failed = [src for src, pr in procs if pr.wait() != 0]
    if failed:
        raise RuntimeError(f"nvcc failed on {failed}")
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call([NVCC, "--shared", "-gencode", "arch=compute_100a,code=sm_100a",
                           "-o", tmp, *objs, "-lcudart_static", "-ldl", "-lrt", "-lpthread"])
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
