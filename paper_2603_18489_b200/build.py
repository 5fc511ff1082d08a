"""Builds libentropycache.so (sm_100a only) and its Python marshalling module in-tree, beside this file.

    python paper_2603_18489_b200/build.py [--force] [--verbose]

(run by path: importing the package loads the library, which may not exist yet)

Each .cu under csrc/ is compiled to an object under _build/ (git-ignored) and
the objects are linked into one shared library with a static CUDA runtime, so
the library needs nothing but the driver at load time (driver entry points
are resolved through the runtime, so it also loads on a machine without one).
csrc/ec_python.cpp becomes _ec_python.so, linked against that library and PyTorch's.
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OBJDIR = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libentropycache.so")
PY_SRC = os.path.join(CSRC, "ec_python.cpp")
PY_LIB = os.path.join(HERE, "_ec_python.so")

NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
ARCH_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a"]
CFLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]


def _newer(target: str, deps: list[str]) -> bool:
    if not os.path.exists(target):
        return False
    t = os.path.getmtime(target)
    return all(os.path.getmtime(d) <= t for d in deps)


def _compile(src: str, verbose: bool) -> str:
    obj = os.path.join(OBJDIR, os.path.basename(src)[:-3] + ".o")
    headers = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h"))
    if _newer(obj, [src] + headers):
        return obj
    cmd = [NVCC] + ARCH_FLAGS + CFLAGS + ["-c", src, "-o", obj]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
        print(" ".join(cmd), flush=True)
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode:
        raise RuntimeError(f"nvcc failed on {src}")
    return obj


def _build_python_module(force: bool, verbose: bool) -> None:
    if not force and _newer(PY_LIB, [PY_SRC] + glob.glob(os.path.join(INCLUDE, "*.h"))):
        return
    import torch                      # for its headers and libraries only
    t = os.path.dirname(torch.__file__)
    tmp = PY_LIB + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", INCLUDE, "-I", sysconfig.get_paths()["include"], "-I", os.path.join(t, "include"),
           "-I", os.path.join(t, "include", "torch", "csrc", "api", "include"),
           "-I", os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include"), PY_SRC, "-o", tmp,
           "-L", HERE, "-l:libentropycache.so", "-L", os.path.join(t, "lib"),
           "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-Wl,-rpath,$ORIGIN"]
    if verbose:
        print(" ".join(cmd), flush=True)
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode:
        raise RuntimeError(f"{cmd[0]} failed on {PY_SRC}")
    os.replace(tmp, PY_LIB)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJDIR, exist_ok=True)
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    if force:
        for o in glob.glob(os.path.join(OBJDIR, "*.o")):
            os.remove(o)
    with cf.ThreadPoolExecutor(max_workers=min(8, len(srcs))) as ex:
        objs = list(ex.map(lambda s: _compile(s, verbose), srcs))
    stale = [o for o in glob.glob(os.path.join(OBJDIR, "*.o")) if o not in objs]
    for o in stale:
        os.remove(o)
    if force or not _newer(LIB, objs):
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [NVCC] + ARCH_FLAGS + ["-shared", "-o", tmp] + objs
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
        os.replace(tmp, LIB)
    _build_python_module(force, verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
