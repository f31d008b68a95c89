"""Compile the CUDA library (sm_100a) into ``libtrdq.so`` and the native part of its binding into ``_calls.<torch>.<python>.so``, next to this file.

nvcc cross-compiles without a GPU, so this runs on a CPU-only machine too.  The
CUDA runtime is linked statically and the driver API is reached through the
runtime at run time, so the shared object loads on a machine without a driver.
``libtrdq.so`` needs nvcc alone; the native calls need torch and a C++ compiler, and where
they are missing the calls are left out with a warning.
"""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libtrdq.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--fmad=false",            # fp32 adds and multiplies stay separately rounded; FMAs are written explicitly
    "-Xcompiler", "-fPIC",
    "-cudart", "static",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def calls_path() -> str:
    """The native calls for the torch and the Python at hand.  They have the class layouts of both compiled in, so the file name says which
    they are: under another torch or Python the file is not found, rather than loaded and wrong."""
    import sysconfig

    import torch
    return os.path.join(HERE, f"_calls.torch-{torch.__version__}-abi{int(torch.compiled_with_cxx11_abi())}.{sysconfig.get_config_var('SOABI')}.so")


def _calls_stale(path: str) -> bool:
    deps = [os.path.join(CSRC, "calls.cpp"), os.path.join(HERE, "..", "include", "trdq.h"), __file__]
    return not os.path.exists(path) or any(os.path.getmtime(d) > os.path.getmtime(path) for d in deps)


def _calls_command(out: str) -> list:
    import sysconfig

    import torch
    base = os.path.dirname(torch.__file__)
    toolkit = os.path.dirname(os.path.dirname(shutil.which(NVCC) or NVCC))   # (NVCC may be a name on PATH)
    include = [os.path.join(base, "include"), os.path.join(base, "include", "torch", "csrc", "api", "include"),
               sysconfig.get_paths()["include"], os.path.join(toolkit, "include")]
    return [os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
            *(f"-I{d}" for d in include), os.path.join(CSRC, "calls.cpp"), "-o", out,
            "-L" + os.path.join(base, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) \
        + [os.path.join(HERE, "..", "include", "trdq.h"), __file__]
    return any(os.path.getmtime(d) > t for d in deps)


def _start_calls(force: bool):
    """The compiler of the native calls at work and what it makes, or None if there is nothing to do or it cannot even be started.  The binding
    does without them (with a warning), so this never keeps the library from being built."""
    try:
        for old in glob.glob(os.path.join(HERE, "_calls*.so")):
            if _calls_stale(old):
                os.remove(old)   # whatever happens next: it was made from other sources, for whichever torch
        path = calls_path()
        if not force and os.path.exists(path):
            return None
        cmd = _calls_command(path + ".new")
        return subprocess.Popen(cmd), cmd, path
    except (ImportError, OSError) as e:
        warnings.warn(f"the native calls of the binding are not built: {e}")
        return None


def _finish_calls(started) -> None:
    if not started:
        return
    process, cmd, path = started
    if process.wait() == 0:
        os.replace(path + ".new", path)
    else:
        warnings.warn("the native calls of the binding are not built, compiler failed: " + " ".join(cmd))


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
    started = _start_calls(force)
    try:
        if force or _stale():
            _build_library(verbose)
    finally:
        _finish_calls(started)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
