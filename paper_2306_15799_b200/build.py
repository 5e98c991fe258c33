"""Builds libflurka.so (the C-ABI CUDA library, nvcc for sm_100a) and _marshal.so (argument marshalling) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libflurka.so")
MARSHAL = os.path.join(HERE, "_marshal.so")
MARSHAL_SOURCE = os.path.join(CSRC, "marshal.cpp")


def sources():
    return [os.path.join(CSRC, f) for f in sorted(os.listdir(CSRC)) if f.endswith(".cu")]


def _deps():
    out = list(sources())
    out += [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    out.append(os.path.join(ROOT, "include", "flurka.h"))
    return out


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(p) > t for p in _deps())


def marshal_tag() -> bytes:
    """What the module is built for: it holds this text."""
    import torch
    return ("marshalling for torch %s, %s" % (torch.__version__, sys.implementation.cache_tag)).encode()


def marshal_fits() -> bool:
    """Whether _marshal.so is there and was built for the torch and the Python that run now."""
    if not os.path.exists(MARSHAL):
        return False
    with open(MARSHAL, "rb") as f:
        return marshal_tag() in f.read()


def compile_marshal(source: str, target: str) -> None:
    """g++ against torch's headers: marshal.cpp -> a Python module"""
    import sysconfig
    import torch
    root = os.path.join(os.path.dirname(os.path.abspath(torch.__file__)))
    tmp = target + ".tmp.%d" % os.getpid()
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-DFLURKA_MARSHAL_TAG=\"%s\"" % marshal_tag().decode(),
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
           "-isystem", os.path.join(root, "include"), "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"),
           "-isystem", os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"),
           "-isystem", sysconfig.get_paths()["include"], source, "-o", tmp,
           "-L", os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("g++ failed building _marshal.so")
    os.replace(tmp, target)


def build_marshal(force: bool = False) -> str:
    """paper_2306_15799_b200/_marshal.so"""
    if force or not marshal_fits() or os.path.getmtime(MARSHAL) < os.path.getmtime(MARSHAL_SOURCE):
        compile_marshal(MARSHAL_SOURCE, MARSHAL)
    return MARSHAL


def build(force: bool = False, verbose: bool = False) -> str:
    """nvcc -gencode arch=compute_100a,code=sm_100a -> paper_2306_15799_b200/libflurka.so (and _marshal.so)"""
    build_marshal(force)
    if not force and not is_stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", tmp]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += sources()
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("nvcc failed building libflurka.so")
    if verbose:
        sys.stderr.write(res.stderr)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
