"""Builds libpyramidkv.so (the C-ABI CUDA library) with nvcc for sm_100a and _pkv_native.so (the native half of the
Python binding) with g++, both in-tree."""
from __future__ import annotations

import glob
import hashlib
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libpyramidkv.so")
STAMP = LIB + ".srchash"      # digest of the sources the library was built from (travels with the library)
BINDING_SRC = os.path.join(PKG, "native", "pkv_bind.cpp")
BINDING = os.path.join(PKG, "_pkv_native.so")
BINDING_FLAGS = ["-O2", "-std=c++17", "-fPIC", "-shared"]
BINDING_LIBS = ["-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-shared"]


def _flags():
    """NVCC_FLAGS plus whatever PKV_NVCC_EXTRA adds (e.g. -DPKV_POLY_PAIRS=4 to move the split of the exponentials)."""
    return NVCC_FLAGS + os.environ.get("PKV_NVCC_EXTRA", "").split()


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def source_digest() -> str:
    """SHA-256 over the names and contents of everything the library is compiled from."""
    h = hashlib.sha256()
    for f in sorted(glob.glob(os.path.join(CSRC, "*")) + glob.glob(os.path.join(ROOT, "include", "*.h"))):
        h.update(os.path.basename(f).encode())
        with open(f, "rb") as fh:
            h.update(fh.read())
    h.update(" ".join(_flags()).encode())
    return h.hexdigest()


def _stale() -> bool:
    """True when the library is missing or was built from other sources.  Compared by content, not by
    modification time: a copy of the tree to another machine does not keep the times in order."""
    if not os.path.exists(LIB) or not os.path.exists(STAMP):
        return True
    with open(STAMP) as fh:
        return fh.read().strip() != source_digest()


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into one shared library.  Returns its path."""
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc] + _flags() + ["-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", tmp] + sources()
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
        print(" ".join(cmd), file=sys.stderr)
    digest = source_digest()
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    with open(STAMP, "w") as fh:
        fh.write(digest + "\n")
    return LIB


def binding_digest() -> str:
    """SHA-256 over what _pkv_native.so is compiled from and against."""
    import torch
    h = hashlib.sha256()
    for f in (BINDING_SRC, os.path.join(ROOT, "include", "pyramidkv.h")):
        with open(f, "rb") as fh:
            h.update(fh.read())
    h.update(" ".join(BINDING_FLAGS + BINDING_LIBS + [torch.__version__, sysconfig.get_python_version()]).encode())
    return h.hexdigest()


def build_binding(force: bool = False) -> str:
    """Compile native/pkv_bind.cpp against torch's headers and libpyramidkv.so (built first).  Returns its path."""
    build_library(force)
    stamp = BINDING + ".srchash"
    digest = binding_digest()
    if not force and os.path.exists(BINDING) and os.path.exists(stamp):
        with open(stamp) as fh:
            if fh.read().strip() == digest:
                return BINDING
    import torch
    home = os.path.dirname(torch.__file__)
    inc = os.path.join(home, "include")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    dirs = [os.path.join(ROOT, "include"), sysconfig.get_paths()["include"], inc,
            os.path.join(inc, "torch", "csrc", "api", "include"), os.path.join(cuda, "include")]
    tmp = BINDING + ".tmp.%d" % os.getpid()
    # torch's libraries are found by name among those the running interpreter has loaded with torch
    subprocess.check_call([os.environ.get("CXX", "g++")] + BINDING_FLAGS + ["-I" + d for d in dirs] +
                          [BINDING_SRC, "-o", tmp, "-L" + PKG, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN",
                           "-L" + os.path.join(home, "lib")] + BINDING_LIBS)
    os.replace(tmp, BINDING)
    with open(stamp, "w") as fh:
        fh.write(digest + "\n")
    return BINDING


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
    print(build_binding())
