"""Compile the CUDA library (sm_100a) into ``libtrdq.so`` and the native part of its binding into ``_calls.so``, next to this file.

nvcc cross-compiles without a GPU, so this runs on a CPU-only machine too.  The
CUDA runtime is linked statically and the driver API is reached through the
runtime at run time, so the shared object loads on a machine without a driver.
``libtrdq.so`` needs nvcc alone; ``_calls.so`` needs torch and a C++ compiler, and where
they are missing it is left out with a warning.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libtrdq.so")
CALLS = os.path.join(HERE, "_calls.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--fmad=false",            # fp32 adds and multiplies stay separately rounded; FMAs are written explicitly
    "-Xcompiler", "-fPIC",
    "-cudart", "static",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _calls_stale() -> bool:
    deps = [os.path.join(CSRC, "calls.cpp"), os.path.join(HERE, "..", "include", "trdq.h"), __file__]
    return not os.path.exists(CALLS) or any(os.path.getmtime(d) > os.path.getmtime(CALLS) for d in deps)


def _calls_command() -> list:
    import sysconfig

    import torch
    base = os.path.dirname(torch.__file__)
    include = [os.path.join(base, "include"), os.path.join(base, "include", "torch", "csrc", "api", "include"),
               sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include")]
    return [os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            *(f"-I{d}" for d in include), os.path.join(CSRC, "calls.cpp"), "-o", CALLS + ".new",
            "-L" + os.path.join(base, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) \
        + [os.path.join(HERE, "..", "include", "trdq.h"), __file__]
    return any(os.path.getmtime(d) > t for d in deps)


def _start_calls():
    """The compiler of the native calls at work, or None if it cannot even be started.  The binding does without them (with a warning), so this never
    keeps the library from being built."""
    try:
        if os.path.exists(CALLS):
            os.remove(CALLS)   # whatever happens next: it was made from other sources
        cmd = _calls_command()
        return subprocess.Popen(cmd), cmd
    except (ImportError, OSError) as e:
        warnings.warn(f"the native calls of the binding are not built: {e}")
        return None


def _finish_calls(started) -> None:
    if not started:
        return
    if started[0].wait() == 0:
        os.replace(CALLS + ".new", CALLS)
    else:
        warnings.warn("the native calls of the binding are not built, compiler failed: " + " ".join(started[1]))


def _build_library(verbose: bool) -> None:
    procs = []
    objs = []
    for src in sources():
        obj = os.path.join(CSRC, os.path.basename(src)[:-3] + ".o")
        cmd = [NVCC, *FLAGS, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((subprocess.Popen(cmd), cmd))
        objs.append(obj)
    for p, cmd in procs:
        if p.wait() != 0:
            raise RuntimeError("nvcc failed: " + " ".join(cmd))
    subprocess.run([NVCC, "-shared", "-cudart", "static", "-o", LIB, *objs], check=True)


def build(force: bool = False, verbose: bool = False) -> str:
    started = _start_calls() if force or _calls_stale() else None
    try:
        if force or _stale():
            _build_library(verbose)
    finally:
        _finish_calls(started)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
