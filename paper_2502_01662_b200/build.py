"""Builds libcos_verify.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the module _call, the call from Python, with g++."""
from __future__ import annotations

import glob
import importlib.metadata
import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB = os.path.join(PKG_DIR, "libcos_verify.so")
CALL_SOURCE = os.path.join(CSRC, "call.cpp")
OBJ_DIR = os.path.join(PKG_DIR, "_build")


def nvcc_path() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; set NVCC or put it on PATH")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def dependencies():
    return sources() + sorted(glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h"))) + [os.path.join(INCLUDE, "cos_verify.h")]


def _stale(path: str, deps) -> bool:
    return not os.path.exists(path) or any(os.path.getmtime(d) > os.path.getmtime(path) for d in deps)


def needs_build() -> bool:
    return _stale(LIB, dependencies())


def call_path() -> str:
    """Where the module of csrc/call.cpp for this interpreter and this torch is: it holds inline code of both, so that one made for others is
    not to be opened.  Raises PackageNotFoundError without torch."""
    return os.path.join(PKG_DIR, "_call.%s.torch-%s.so" % (sysconfig.get_config_var("SOABI"), importlib.metadata.version("torch")))


def call_needs_build() -> bool:
    return _stale(call_path(), [CALL_SOURCE, os.path.join(INCLUDE, "cos_verify.h")])


def _compile(src: str, verbose: bool):
    obj = os.path.join(OBJ_DIR, os.path.splitext(os.path.basename(src))[0] + ".o")
    cmd = [
        nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
        "-Xptxas", "-v" if verbose else "-O3", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC, "-c", "-o", obj, src,
    ]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + res.stdout + res.stderr)
    return obj, res.stdout + res.stderr


def _compile_call(out: str):
    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda = os.path.join(os.path.dirname(os.path.dirname(nvcc_path())), "include")
    cmd = ["g++", "-O2", "-std=c++20", "-fPIC", "-shared", "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI, "-I", INCLUDE, "-isystem", inc,
           "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"), "-isystem", cuda, "-isystem", sysconfig.get_paths()["include"], "-o", out,
           CALL_SOURCE, "-L", lib, "-Wl,-rpath," + lib, "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("g++ failed:\n" + " ".join(cmd) + "\n" + res.stdout + res.stderr)


def build_call(force: bool = False) -> str:
    """Compile the module of csrc/call.cpp if there is none for this interpreter and this torch, or an older one; return its path."""
    path = call_path()
    if force or call_needs_build():
        fresh = "%s.%d" % (path, os.getpid())
        _compile_call(fresh)
        os.replace(fresh, path)  # (another process may be at it too)
    return path


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile the CUDA library if it is missing or older than its sources; return its path.
    Every csrc/*.cu is one translation unit; they are compiled side by side and linked into one library."""
    if not force and not needs_build():
        return LIB
    os.makedirs(OBJ_DIR, exist_ok=True)
    srcs = sources()
    with ThreadPoolExecutor(max_workers=len(srcs)) as pool:
        done = list(pool.map(lambda s: _compile(s, verbose), srcs))
    cmd = [nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-Xcompiler", "-fPIC", "-o", LIB]
    cmd += [obj for obj, _ in done] + ["-lcudart"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("link failed:\n" + " ".join(cmd) + "\n" + res.stdout + res.stderr)
    if verbose:
        for _, log in done:
            sys.stderr.write(log)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
    print(build_call(force=True))
