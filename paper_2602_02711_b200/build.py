"""Builds libdmr.so in-tree with nvcc for sm_100a (cross-compiles without a GPU).

Every .cu file is compiled to an object of its own (in parallel, only when it or a header changed)
and the objects are linked into the shared library.  csrc/calls.cpp becomes the extension module _calls.so beside it.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor
from importlib import metadata

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libdmr.so")
CALLS_SRC = os.path.join(CSRC, "calls.cpp")
CALLS = os.path.join(PKG, "_calls.so")
CALLS_STAMP = os.path.join(OBJ, "calls.txt")  # what CALLS was built for

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC,
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def headers():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))


def _obj(src: str) -> str:
    return os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _calls_made_for() -> str:
    return f"torch {metadata.version('torch')}, Python {sys.version_info[0]}.{sys.version_info[1]}"


def _calls_stale() -> bool:
    # the module is bound to the torch and Python it was built with, whatever the files' times say
    try:
        with open(CALLS_STAMP) as f:
            made_for = f.read()
    except OSError:
        return True
    return made_for != _calls_made_for() or _stale(CALLS, [CALLS_SRC] + headers())


def needs_build() -> bool:
    return _stale(LIB, sources() + headers()) or _calls_stale()


def _calls_command() -> list:
    import torch  # for its paths
    base = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            "-I" + os.path.join(ROOT, "include"), "-I" + sysconfig.get_paths()["include"], "-I" + os.path.join(cuda, "include"),
            "-I" + os.path.join(base, "include"), CALLS_SRC, "-o", CALLS, "-L" + os.path.join(base, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ, exist_ok=True)
    hdrs = headers()
    todo = [s for s in sources() if force or _stale(_obj(s), [s] + hdrs)]

    def compile_one(src):
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", _obj(src)]
        r = subprocess.run(cmd, capture_output=True, text=True)
        return src, r

    calls = subprocess.Popen(_calls_command()) if force or _calls_stale() else None
    with ThreadPoolExecutor(max_workers=min(8, max(1, len(todo)))) as pool:
        for src, r in pool.map(compile_one, todo):
            if verbose or r.returncode != 0:
                sys.stderr.write(r.stdout + r.stderr)
            if r.returncode != 0:
                raise subprocess.CalledProcessError(r.returncode, f"nvcc {src}")
    objs = [_obj(s) for s in sources()]
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "--shared", "-o", LIB] + objs, check=True)
    if calls is not None:
        if calls.wait() != 0:
            raise subprocess.CalledProcessError(calls.returncode, f"{calls.args[0]} {CALLS_SRC}")
        with open(CALLS_STAMP, "w") as f:
            f.write(_calls_made_for())
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
