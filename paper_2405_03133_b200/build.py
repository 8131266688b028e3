"""Builds liblory.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _torch_glue.so (the torch side of
layer.py) with g++ against the installed torch.

    python -m paper_2405_03133_b200.build [--force] [-v] [--debug]
"""
from __future__ import annotations

import hashlib
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liblory.so")
GLUE_SRC = os.path.join(HERE, "csrc_torch", "glue.cpp")
GLUE = os.path.join(HERE, "_torch_glue.so")         # the torch side of layer.py (g++, no device code)
LIB_DEBUG = os.path.join(HERE, "liblory_debug.so")   # the same sources with -DLORY_DEBUG (bounds checks in the kernels)
SOURCES = ["lory_api.cu", "routing.cu", "simt.cu", "tc.cu", "noalloc.cu", "block.cu", "probe.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared",
]


def _stale(lib) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = [os.path.join(CSRC, n) for n in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "lory.h")]
    return any(os.path.getmtime(p) > t for p in deps)


def glue_tag() -> str:
    """What the glue was built from: its sources, the C ABI it calls and the torch it is linked to."""
    import torch
    h = hashlib.sha256(torch.__version__.encode())
    for path in (GLUE_SRC, os.path.join(ROOT, "include", "lory.h")):
        with open(path, "rb") as f:
            h.update(f.read())
    return "lory-glue-" + h.hexdigest()


def glue_is_current() -> bool:
    """Whether _torch_glue.so carries the tag of the sources (asked of the file: a module once loaded cannot be replaced)."""
    if not os.path.exists(GLUE) or not os.path.exists(GLUE_SRC):
        return os.path.exists(GLUE)     # without sources there is nothing to compare with
    with open(GLUE, "rb") as f:
        return glue_tag().encode() in f.read()


def build_glue(force: bool = False) -> str:
    if not force and glue_is_current():
        return GLUE
    import sysconfig

    import torch
    from torch.utils import cpp_extension

    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    inc = cpp_extension.include_paths() + [sysconfig.get_paths()["include"], os.path.join(cuda, "include"),
                                           os.path.join(ROOT, "include")]
    libdir = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = f"{GLUE}.{os.getpid()}"      # moved into place: another process may be importing the module
    cmd = ([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-DTORCH_EXTENSION_NAME=_torch_glue",
            f'-DLORY_GLUE_TAG="{glue_tag()}"', f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"] + ["-I" + p for p in inc] + [GLUE_SRC] +
           ["-L" + libdir, "-Wl,-rpath," + libdir, "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python", "-lc10",
            "-lc10_cuda", "-ldl", "-o", tmp])
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("g++ failed:\n" + res.stdout + res.stderr)
    os.replace(tmp, GLUE)
    return GLUE


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    lib = LIB_DEBUG if debug else LIB
    if not force and not _stale(lib):
        return lib
    nvcc = os.environ.get("NVCC", "nvcc")
    cmd = [nvcc] + NVCC_FLAGS + ["-I" + os.path.join(ROOT, "include"), "-I" + CSRC]
    if debug:
        cmd += ["-DLORY_DEBUG"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", lib]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    if verbose:
        print(res.stderr)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug="--debug" in sys.argv))
    print(build_glue(force="--force" in sys.argv))
