"""Builds libagileq.so (nvcc, sm_100a; cross-compiles without a GPU) and the binding's native half in-tree.

The library needs nvcc and its host compiler only (`build_library`); the native half of the Python binding also needs the
C++ headers and libraries of this interpreter and its torch. Environment: NVCC, CXX."""
from __future__ import annotations

import glob
import importlib.metadata
import os
import shutil
import subprocess
import sys
import sysconfig

_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_DIR, "csrc")
LIB = os.path.join(_DIR, "libagileq.so")
# native half of the binding: a CPython module against this interpreter's torch, linked to the library beside it
HOST_SRC = os.path.join(CSRC, "aq_host.cpp")
HOST_LIB = os.path.join(_DIR, "_aq_host.so")
HOST_TAG = os.path.join(_DIR, "_aq_host.built_for")           # the interpreter and torch it was built for

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC", "-Xptxas", "-v",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        [os.path.join(os.path.dirname(_DIR), "include", "agileq.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _nvcc() -> str:
    return os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def _host_tag() -> str:
    return f"{sys.implementation.cache_tag} {sysconfig.get_platform()} torch {importlib.metadata.version('torch')}"


def _host_stale() -> bool:
    header = os.path.join(os.path.dirname(_DIR), "include", "agileq.h")
    if not os.path.exists(HOST_LIB) or os.path.getmtime(HOST_LIB) < max(os.path.getmtime(HOST_SRC), os.path.getmtime(header)):
        return True
    if not os.path.exists(HOST_TAG):
        return True
    with open(HOST_TAG) as f:
        return f.read() != _host_tag()


def _build_host() -> None:
    import torch
    root = os.path.dirname(torch.__file__)
    nvcc = os.path.realpath(shutil.which(_nvcc()) or _nvcc())
    python, cuda = sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    for header in (os.path.join(python, "Python.h"), os.path.join(root, "include", "ATen", "ATen.h"),
                   os.path.join(cuda, "cuda_runtime_api.h")):
        if not os.path.exists(header):
            raise RuntimeError(f"{LIB} is built; the Python binding beside it needs {header}, which is missing")
    tmp = HOST_LIB + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", HOST_SRC, "-o", tmp,
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
           "-I" + python, "-I" + os.path.join(root, "include"),
           "-I" + os.path.join(root, "include", "torch", "csrc", "api", "include"), "-I" + cuda,
           "-L" + os.path.join(root, "lib"), "-Wl,-rpath," + os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu",
           "-ltorch_python", "-L" + _DIR, "-l:libagileq.so", "-Wl,-rpath,$ORIGIN"]
    subprocess.check_call(cmd)
    os.replace(tmp, HOST_LIB)
    with open(HOST_TAG, "w") as f:
        f.write(_host_tag())


def build(force: bool = False, verbose: bool = False) -> str:
    lib = build_library(force, verbose)
    if force or _host_stale():
        _build_host()
    return lib


def build_library(force: bool = False, verbose: bool = False) -> str:
    """The C library alone."""
    if not force and not _stale():
        return LIB
    nvcc = _nvcc()
    objs = []
    procs = []
    for src in sources():
        obj = src[:-3] + ".o"
        objs.append(obj)
        procs.append((src, subprocess.Popen([nvcc, *NVCC_FLAGS, "-c", src, "-o", obj],
                                            stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    log = []
    for src, p in procs:
        out, _ = p.communicate()
        log.append(out)
        if p.returncode != 0:
            sys.stderr.write(out)
            raise RuntimeError(f"nvcc failed on {src}")
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.check_call([nvcc, "-shared", "-o", tmp, *objs, "-lcudart_static", "-lpthread", "-ldl", "-lrt"])
    os.replace(tmp, LIB)
    with open(os.path.join(_DIR, "build.log"), "w") as f:
        f.write("\n".join(log))
    if verbose:
        print("\n".join(log))
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
