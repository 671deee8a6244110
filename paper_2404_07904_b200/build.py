"""Builds the C-ABI shared library in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the extension module
that marshals torch tensors into it with the host compiler."""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
CSRC = os.path.join(_PKG, "csrc")
LIB = os.path.join(_PKG, "libhgrn2.so")
MARSHAL_SRC = os.path.join(_PKG, "native", "marshal.cpp")
MARSHAL = os.path.join(_PKG, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
    "-shared", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in deps)


def _headers():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(_ROOT, "include", "*.h"))


def build_marshal(force: bool = False) -> str:
    """Compile native/marshal.cpp against the installed torch (its headers only; nothing is generated)."""
    if not force and not _stale(MARSHAL, [MARSHAL_SRC, os.path.join(_ROOT, "include", "hgrn2.h")]):
        return MARSHAL
    import torch
    top = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    tmp = MARSHAL + ".tmp.%d" % os.getpid()
    subprocess.check_call(
        [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
         "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch.compiled_with_cxx11_abi(), "-I", os.path.join(_ROOT, "include"),
         "-isystem", os.path.join(top, "include"), "-isystem", os.path.join(top, "include", "torch", "csrc", "api", "include"),
         "-isystem", os.path.join(cuda, "include"), "-isystem", sysconfig.get_paths()["include"], MARSHAL_SRC, "-o", tmp,
         "-L" + _PKG, "-l:libhgrn2.so", "-L" + os.path.join(top, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10",
         "-lc10_cuda", "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, MARSHAL)
    return MARSHAL


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into libhgrn2.so (only when a source is newer than the library), then the
    marshalling module."""
    if not force and not _stale(LIB, sources() + _headers()):
        build_marshal()
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc] + NVCC_FLAGS + ["-I", os.path.join(_ROOT, "include"), "-I", CSRC]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += ["-o", tmp] + sources()
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    build_marshal(force)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
