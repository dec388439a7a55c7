"""Builds ``libvitcop.so`` (sm_100a, nvcc) and the Python caller (``_call.<interpreter>-<machine>-torch<version>.so``, g++) in-tree.
``python -m paper_2601_17818_b200.build``."""
from __future__ import annotations

import concurrent.futures as cf
import hashlib
import os
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD_DIR = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libvitcop.so")
SOURCES = ["api.cu", "knorm.cu", "select.cu", "compact.cu", "filter.cu", "gram.cu", "density.cu", "nearest.cu", "kproj.cu", "merge.cu", "saliency.cu",
           "schedule.cu"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
              "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _digest() -> str:
    h = hashlib.sha1(" ".join(NVCC_FLAGS).encode())
    for name in sorted(set(os.listdir(CSRC)) - {"call.cpp"}) + ["../../include/vitcop.h"]:
        with open(os.path.join(CSRC, name), "rb") as fh:
            h.update(name.encode() + fh.read())
    return h.hexdigest()


def caller_path() -> str:
    """The Python caller built for this interpreter and torch: it is compiled against both, so their versions are in its name and
    one built for others is not found."""
    import platform

    import torch
    return os.path.join(PKG, f"_call.{sys.implementation.cache_tag}-{platform.machine()}-torch{torch.__version__}.so")


def _caller_flags() -> list:
    import torch
    return ["-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            "-lc10", "-ltorch_cpu", "-ltorch_python"]


def _caller_digest() -> str:
    """Of what the caller is made of: sources, flags, and the torch and the interpreter whose headers it is compiled against."""
    import torch
    h = hashlib.sha1(" ".join([*_caller_flags(), torch.__version__, sys.implementation.cache_tag]).encode())
    for name in (os.path.join(CSRC, "call.cpp"), os.path.join(INCLUDE, "vitcop.h")):
        with open(name, "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()


def build_caller(force: bool = False) -> str:
    """A CPython extension that unpacks torch tensors (headers of the torch that imports it); returns its path."""
    import sysconfig

    import torch
    from torch.utils import cpp_extension
    path, dig = caller_path(), _caller_digest()
    stamp = os.path.join(BUILD_DIR, os.path.basename(path) + ".stamp")
    if not force and os.path.exists(path) and os.path.exists(stamp) and open(stamp).read() == dig:
        return path
    os.makedirs(BUILD_DIR, exist_ok=True)
    inc = [a for p in [*cpp_extension.include_paths(), sysconfig.get_paths()["include"], INCLUDE] for a in ("-I", p)]
    flags, tmp = _caller_flags(), path + f".tmp{os.getpid()}"
    cmd = ["g++", *(f for f in flags if not f.startswith("-l")), *inc, os.path.join(CSRC, "call.cpp"), "-o", tmp,
           "-L", os.path.join(os.path.dirname(torch.__file__), "lib"), *(f for f in flags if f.startswith("-l"))]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode:
        sys.stderr.write(f"$ {' '.join(cmd)}\n{r.stdout}{r.stderr}")
        raise RuntimeError("g++ failed on call.cpp")
    os.replace(tmp, path)
    with open(stamp, "w") as fh:
        fh.write(dig)
    return path


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every translation unit for sm_100a and link the shared library, and the Python caller; returns the library's path."""
    os.makedirs(BUILD_DIR, exist_ok=True)
    stamp = os.path.join(BUILD_DIR, "stamp")
    dig = _digest()
    if not force and os.path.exists(LIB) and os.path.exists(stamp) and open(stamp).read() == dig:
        build_caller()
        return LIB

    def compile_one(src: str) -> str:
        obj = os.path.join(BUILD_DIR, src.replace(".cu", ".o"))
        cmd = [_nvcc(), *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode:
            sys.stderr.write(f"$ {' '.join(cmd)}\n{r.stdout}{r.stderr}")
        if r.returncode:
            raise RuntimeError(f"nvcc failed on {src}")
        return obj

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES) + 1) as ex:
        caller = ex.submit(build_caller, force)
        objs = list(ex.map(compile_one, SOURCES))
        caller.result()
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.check_call([_nvcc(), "-shared", "-gencode", "arch=compute_100a,code=sm_100a", *objs, "-o", tmp])
    os.replace(tmp, LIB)
    with open(stamp, "w") as fh:
        fh.write(dig)
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
