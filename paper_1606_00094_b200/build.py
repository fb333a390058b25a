"""Builds the CUDA library (``libboda.so``) in-tree with nvcc for sm_100a, and with g++ the extension through which the
binding calls it with torch tensors (``_torch_calls-<python>-<torch>.so``).

    python -m paper_1606_00094_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import glob
import importlib.metadata
import os
import shutil
import subprocess
import sys
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
CSRC = os.path.join(_PKG, "csrc")
LIB_PATH = os.path.join(_PKG, "libboda.so")
CALLS_SRC = os.path.join(CSRC, "torch_calls.cpp")
CALLS_HEADER = os.path.join(_ROOT, "include", "boda.h")
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-shared"] + os.environ.get("BODA_NVCC_EXTRA", "").split()


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: cannot build libboda.so")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def is_stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    deps = sources() + _headers()
    return any(os.path.getmtime(p) > t for p in deps)


def _headers():
    return glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) \
        + glob.glob(os.path.join(_ROOT, "include", "*.h"))


def calls_path():
    """Where the extension for this Python and the installed torch lies (None: no torch).  It is bound to the C++ interfaces of both, so
    another version of either looks for another file."""
    try:
        version = importlib.metadata.version("torch")
    except importlib.metadata.PackageNotFoundError:
        return None
    return os.path.join(_PKG, f"_torch_calls-{sys.implementation.cache_tag}-torch{version}.so")


def calls_stale() -> bool:
    path = calls_path()
    return path is not None and (not os.path.exists(path) or
                                 os.path.getmtime(path) <= max(os.path.getmtime(p) for p in (CALLS_SRC, CALLS_HEADER)))


def build_calls(force: bool = False):
    """Compile the extension over torch tensors; returns its path (None without torch: the library serves raw addresses)."""
    path = calls_path()
    if path is None or not (force or calls_stale()):
        return path
    import torch
    from torch.utils import cpp_extension
    tmp = path + f".tmp{os.getpid()}"
    cuda_home = os.path.dirname(os.path.dirname(_nvcc()))
    includes = [sysconfig.get_paths()["include"], *cpp_extension.include_paths(), os.path.join(cuda_home, "include")]
    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    cmd += [a for i in includes for a in ("-isystem", i)] + ["-I", os.path.dirname(CALLS_HEADER), "-o", tmp, CALLS_SRC, "-L", libs]
    res = subprocess.run(cmd + ["-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"], capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("g++ failed:\n" + res.stdout + res.stderr)
    os.replace(tmp, path)
    for old in glob.glob(os.path.join(_PKG, "_torch_calls*.so")):
        if old != path:
            os.remove(old)
    return path


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every ``csrc/*.cu`` into one shared library; returns its path.

    Each source is compiled to an object under ``csrc/build/`` (in parallel, and only if it or a header changed),
    then the objects are linked."""
    build_calls(force)
    if not force and not is_stale():
        return LIB_PATH
    nvcc = _nvcc()
    objdir = os.path.join(CSRC, "build")
    os.makedirs(objdir, exist_ok=True)
    hdr_time = max(os.path.getmtime(h) for h in _headers())
    compile_flags = [f for f in NVCC_FLAGS if f != "-shared"]
    jobs, objs = [], []
    for src in sources():
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if not force and os.path.exists(obj) and os.path.getmtime(obj) > max(os.path.getmtime(src), hdr_time):
            continue
        cmd = [nvcc] + compile_flags + (["-Xptxas", "-v"] if verbose else []) + \
              ["-I", CSRC, "-I", os.path.join(_ROOT, "include"), "-c", "-o", obj, src]
        jobs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    log = []
    failed = False
    for src, proc in jobs:
        out, _ = proc.communicate()
        log.append(out)
        if proc.returncode != 0:
            failed = True
    if failed:
        raise RuntimeError("nvcc failed:\n" + "".join(log))
    if verbose:
        print("".join(log))
    tmp = LIB_PATH + f".tmp{os.getpid()}"
    res = subprocess.run([nvcc, "-shared", "-o", tmp] + objs, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("link failed:\n" + res.stdout + res.stderr)
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
