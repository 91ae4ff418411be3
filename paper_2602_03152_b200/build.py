"""Builds `libfasa.so` (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and `_marshal.so` (the
argument marshalling of the Python binding) with the host compiler.

    python -m paper_2602_03152_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import glob
import importlib.metadata
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libfasa.so")
MARSHAL_SRC = os.path.join(CSRC, "marshal.cpp")
MARSHAL = os.path.join(PKG, "_marshal.so")

NVCC_FLAGS = [
    "-std=c++17", "-O3", "-lineinfo",
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-Xcompiler", "-fPIC", "-shared", "-cudart", "static", "--threads", "0",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > os.path.getmtime(LIB) for d in deps)


def marshal_tag() -> str:
    """The interpreter and torch that an extension module built now is for; a string that the file holds."""
    return "_marshal for %s, torch %s" % (sysconfig.get_config_var("SOABI"), importlib.metadata.version("torch"))


def marshal_fits(path: str) -> bool:
    """Whether the extension module at `path` was built for this interpreter and this torch."""
    with open(path, "rb") as f:
        return marshal_tag().encode() in f.read()


def _marshal_stale() -> bool:
    return not os.path.exists(MARSHAL) or os.path.getmtime(MARSHAL_SRC) > os.path.getmtime(MARSHAL) or not marshal_fits(MARSHAL)


def build_marshal(force: bool = False) -> str:
    """The binding's extension module, against the headers and libraries of the installed torch."""
    if not force and not _marshal_stale():
        return MARSHAL
    import torch

    root = os.path.dirname(torch.__file__)
    libs = os.path.join(root, "lib")
    tmp = MARSHAL + ".tmp.%d" % os.getpid()
    cmd = ["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI,
           '-DFASA_BUILT_FOR="%s"' % marshal_tag()]
    for path in (sysconfig.get_paths()["include"], "/usr/local/cuda/include"):
        cmd += ["-I", path]
    for path in ("include", os.path.join("include", "torch", "csrc", "api", "include")):
        cmd += ["-isystem", os.path.join(root, path)]
    cmd += ["-o", tmp, MARSHAL_SRC, "-L", libs, "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python",
            "-Wl,-rpath," + libs]
    subprocess.check_call(cmd)
    os.replace(tmp, MARSHAL)
    return MARSHAL


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every kernel into one shared object, and the binding's extension; returns the former's path."""
    marshal = subprocess.Popen([sys.executable, os.path.abspath(__file__), "--marshal"] + (["--force"] if force else [])) \
        if force or _marshal_stale() else None
    if force or _stale():
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        tmp = LIB + ".tmp.%d" % os.getpid()
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
              ["-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", tmp] + sources()
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    if marshal is not None and marshal.wait() != 0:
        raise RuntimeError("building %s failed" % MARSHAL)
    return LIB


if __name__ == "__main__":
    if "--marshal" in sys.argv:
        build_marshal(force="--force" in sys.argv)
    else:
        print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
