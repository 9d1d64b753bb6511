"""Compile the CUDA library (sm_100a only) into paper_2411_00288_b200/libssconv.so, and its CPython binding beside it."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(_HERE)
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libssconv.so")
SOURCES = ["api.cu", "mask.cu", "pool.cu", "depthwise.cu", "train.cu", "wgrad.cu", "forward.cu"]
HEADERS = ["launch.cuh", "layout.cuh", "sm100_ptx.cuh"]


def _newest_source_mtime() -> float:
    files = [os.path.join(CSRC, f) for f in SOURCES + HEADERS] + [os.path.join(ROOT, "include", "ssconv.h")]
    return max(os.path.getmtime(f) for f in files)


def binding_path() -> str:
    """The native binding's file.  It holds for one torch (whose C++ interface is no stable one) and one interpreter, so
    both are part of its name: after a change of either another file is built and looked for."""
    import torch
    return os.path.join(_HERE, f"_binding.torch-{torch.__version__}{sysconfig.get_config_var('EXT_SUFFIX')}")


def build_binding(force: bool = False) -> str:
    """The binding (csrc/binding.cpp) against the installed torch; after the library, which it is linked with."""
    binding = binding_path()
    sources = [os.path.join(CSRC, "binding.cpp"), os.path.join(ROOT, "include", "ssconv.h")]
    if not force and os.path.exists(binding) and os.path.getmtime(binding) >= max(os.path.getmtime(f) for f in sources):
        return binding
    import torch
    t = os.path.dirname(torch.__file__)
    includes = [os.path.join(ROOT, "include"), sysconfig.get_paths()["include"], os.path.join(t, "include"),
                os.path.join(t, "include", "torch", "csrc", "api", "include"),
                os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")]
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC"] + ["-I" + i for i in includes] +
                   [sources[0], "-o", binding, "-L" + os.path.join(t, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu",
                    "-lc10", "-lc10_cuda", "-L" + _HERE, "-l:libssconv.so", "-Wl,-rpath,$ORIGIN"], check=True)
    return binding


def build(force: bool = False, verbose: bool = False) -> str:
    _build_library(force, verbose)
    build_binding(force)
    return LIB


def _build_library(force: bool, verbose: bool) -> str:
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_source_mtime():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-cudart", "static",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", LIB]
    subprocess.run(cmd, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
