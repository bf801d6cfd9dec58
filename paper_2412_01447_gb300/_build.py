"""Builds ``libpldp.so`` in-tree from ``csrc/*.cu`` with nvcc for sm_103a only.

Translation units compile in parallel; the shared library links the CUDA
runtime statically, so it loads without a GPU (the runtime opens the driver at
the first CUDA call).
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import shutil
import subprocess
import sysconfig
import warnings

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB = os.path.join(PKG, "libpldp.so")
CALLS_SRC = os.path.join(CSRC, "host_calls.cpp")
BUILD_DIR = os.path.join(PKG, "_build")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-fvisibility=hidden",
              "-I", INCLUDE, "-I", CSRC]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libpldp.so")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h")) + [
        os.path.abspath(__file__)]


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(p) <= t for p in _deps())


def calls_path() -> str:
    """The binding's native calls, by the torch and the Python that they are for: the
    extension reads tensors through accessors compiled into it, so one built against
    another torch would read their fields in the wrong places."""
    import torch
    return os.path.join(PKG, f"_pldp_calls.torch{torch.__version__}-cxx{int(torch._C._GLIBCXX_USE_CXX11_ABI)}"
                             f"{sysconfig.get_config_var('EXT_SUFFIX')}")


def build_calls(force: bool = False, out: str | None = None, extra_flags=()) -> str:
    """The binding's native checks and marshalling: a Python extension against the
    installed torch's headers and libraries (host code only).  A test build goes to
    another `out` with extra compiler flags."""
    out = out or calls_path()
    deps = [CALLS_SRC, os.path.join(INCLUDE, "pldp.h"), os.path.abspath(__file__)]
    if not force and os.path.exists(out) and all(os.path.getmtime(p) <= os.path.getmtime(out) for p in deps):
        return out
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(nvcc())))
    os.makedirs(os.path.dirname(out), exist_ok=True)
    tmp = out + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *extra_flags,
           "-I", INCLUDE, "-I", os.path.join(root, "include"),
           "-I", os.path.join(root, "include", "torch", "csrc", "api", "include"),
           "-I", sysconfig.get_paths()["include"], "-I", os.path.join(cuda, "include"), CALLS_SRC, "-o", tmp,
           "-L", os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"building the binding's native calls failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, out)
    return out


def _build_calls_if_possible(force: bool = False) -> None:
    """build_calls where a C++ compiler and the headers of torch and Python are found; the
    ctypes form of every call needs none of them."""
    try:
        build_calls(force)
    except Exception as e:
        if os.path.exists(calls_path()):
            os.remove(calls_path())                   # stale: of another state of the sources
        warnings.warn(f"the binding's calls go through ctypes: {e}", RuntimeWarning, stacklevel=2)


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    if not force and up_to_date():
        _build_calls_if_possible()
        return LIB
    os.makedirs(BUILD_DIR, exist_ok=True)
    cc = nvcc()
    objs = []

    def compile_one(src):
        obj = os.path.join(BUILD_DIR, os.path.basename(src)[:-3] + ".o")
        cmd = [cc, *ARCH, *NVCC_FLAGS, *extra_flags, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {os.path.basename(src)}:\n{r.stdout}\n{r.stderr}")
        if verbose and (r.stdout or r.stderr):
            print(r.stdout + r.stderr)
        return obj

    with cf.ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 1)) as ex:
        calls = ex.submit(_build_calls_if_possible, force)
        objs = list(ex.map(compile_one, sources()))
        calls.result()
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [cc, *ARCH, "-shared", "-Xcompiler", "-fPIC", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


def build_variant(name: str, srcs, extra_flags=(), force: bool = False) -> str:
    """Builds a separate shared library ``_build/<name>/lib<name>.so`` from some of
    the sources with extra compiler flags (a test build of selected kernels, e.g.
    with a test-only macro defined).  The product library is not touched."""
    out_dir = os.path.join(BUILD_DIR, name)
    out = os.path.join(out_dir, f"lib{name}.so")
    paths = [os.path.join(CSRC, x) for x in srcs]
    deps = paths + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h")) + [
        os.path.abspath(__file__)]
    if not force and os.path.exists(out) and all(os.path.getmtime(p) <= os.path.getmtime(out) for p in deps):
        return out
    os.makedirs(out_dir, exist_ok=True)
    cc = nvcc()

    def compile_one(src):
        obj = os.path.join(out_dir, os.path.basename(src)[:-3] + ".o")
        r = subprocess.run([cc, *ARCH, *NVCC_FLAGS, *extra_flags, "-c", src, "-o", obj], capture_output=True,
                           text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {os.path.basename(src)}:\n{r.stdout}\n{r.stderr}")
        return obj

    with cf.ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 1)) as ex:
        objs = list(ex.map(compile_one, paths))
    tmp = out + f".tmp{os.getpid()}"
    r = subprocess.run([cc, *ARCH, "-shared", "-Xcompiler", "-fPIC", "-o", tmp, *objs], capture_output=True,
                       text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, out)
    return out
