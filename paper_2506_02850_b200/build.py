"""Builds the CUDA library in-tree: csrc/*.cu -> lib/libmetok.so (sm_100a only), and the native half of
binding.py: csrc/host/calls.cpp -> lib/_metok_calls.so.

nvcc cross-compiles without a GPU, so this runs on any box with the CUDA toolkit.
"""

from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
LIBDIR = os.path.join(PKG, "lib")
OBJDIR = os.path.join(PKG, "_build")
LIB = os.path.join(LIBDIR, "libmetok.so")
# the same sources with short device-side waits, a host switch that withholds one copy, and range checks
# on every data-dependent index: exercises the time-out and unwind paths a normal run never reaches
DEBUG_LIB = os.path.join(LIBDIR, "libmetok_debug.so")
CALLS_SRC = os.path.join(CSRC, "host", "calls.cpp")
CALLS_LIB = os.path.join(LIBDIR, "_metok_calls.so")
DEBUG_DEFINES = ["-DMETOK_DEBUG_SHORT_WAIT", "-DMETOK_DEBUG_BOUNDS"]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
    "--expt-relaxed-constexpr", "--expt-extended-lambda",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build_calls(force: bool = False, verbose: bool = False) -> str:
    """Builds lib/_metok_calls.so against the installed torch."""
    os.makedirs(LIBDIR, exist_ok=True)
    header = os.path.join(os.path.dirname(PKG), "include", "metok.h")
    if force or _stale(CALLS_LIB, [CALLS_SRC, header]):
        from torch.utils import cpp_extension
        cuda = os.path.dirname(os.path.dirname(_nvcc())) if os.path.isabs(_nvcc()) else "/usr/local/cuda"
        includes = [sysconfig.get_paths()["include"], os.path.join(cuda, "include")] + cpp_extension.include_paths()
        cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden"]
        for d in includes:
            cmd += ["-isystem", d]
        cmd += [CALLS_SRC, "-o", CALLS_LIB]
        for d in cpp_extension.library_paths():
            cmd += ["-L", d]
        cmd += ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch", "-ltorch_python"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError("compiling the native calls failed: " + " ".join(cmd))
    return CALLS_LIB


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False, debug: bool = False) -> str:
    """Builds lib/libmetok.so and lib/_metok_calls.so, or with debug=True lib/libmetok_debug.so (see DEBUG_DEFINES)."""
    objdir = OBJDIR + ("_debug" if debug else "")
    lib = DEBUG_LIB if debug else LIB
    defines = DEBUG_DEFINES if debug else []
    os.makedirs(LIBDIR, exist_ok=True)
    os.makedirs(objdir, exist_ok=True)
    nvcc = _nvcc()
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(os.path.dirname(PKG), "include", "metok.h"))
    jobs = []
    objs = []
    for src in sources():
        s = os.path.join(CSRC, src)
        o = os.path.join(objdir, src[:-3] + ".o")
        objs.append(o)
        if force or _stale(o, [s] + headers):
            cmd = [nvcc] + NVCC_FLAGS + defines + (["-Xptxas", "-v"] if ptxas_info else []) + ["-c", s, "-o", o]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        return cmd, r

    with ThreadPoolExecutor(max_workers=min(8, max(1, len(jobs)))) as ex:
        for cmd, r in ex.map(run, jobs):
            if verbose or ptxas_info or r.returncode != 0:
                sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
            if r.returncode != 0:
                raise RuntimeError("nvcc failed: " + " ".join(cmd))
    if force or jobs or _stale(lib, objs):
        cmd = [nvcc, "-shared", "-o", lib] + objs + ["-gencode", "arch=compute_100a,code=sm_100a",
                                                     "-Xcompiler", "-fPIC", "-lcudart_static", "-ldl", "-lrt", "-lpthread"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
    if not debug:
        build_calls(force, verbose)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv, debug="--debug" in sys.argv))
