"""Builds libvocabtrim.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _vt_bind.so (the argument marshalling of the
Python binding) with the C++ compiler against torch's headers.

Usage: python -m paper_2506_22694_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libvocabtrim.so")
OBJ_DIR = os.path.join(HERE, "_build")
BIND_SRC = os.path.join(CSRC, "vt_bind.cpp")
BIND = os.path.join(HERE, "_vt_bind.so")
LIB_STAMPS = os.path.join(HERE, "libvocabtrim_stamps.so")     # -DVT_STAMPS: phase stamps in the head kernel
OBJ_DIR_STAMPS = os.path.join(HERE, "_build_stamps")

NVCC_FLAGS = [
    "-O3", "-std=c++17", "-lineinfo",
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-Xcompiler", "-fPIC",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return _sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))


def needs_build(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    return any(os.path.getmtime(p) > t for p in _deps())


def bind_for() -> str:
    """The Python and torch that an extension module built now is for."""
    import torch

    return "%s, torch %s, C++ ABI %d" % (sys.implementation.cache_tag, torch.__version__, torch._C._GLIBCXX_USE_CXX11_ABI)


def bind_fresh() -> bool:
    """Whether the module is younger than its sources and says that it was built for this Python and torch."""
    newest = max(os.path.getmtime(p) for p in (BIND_SRC, os.path.join(ROOT, "include", "vocabtrim.h")))
    if not os.path.exists(BIND) or os.path.getmtime(BIND) <= newest:
        return False
    with open(BIND, "rb") as f:
        return b"_vt_bind for " + bind_for().encode() + b"\0" in f.read()


def build_bind(force: bool = False) -> str:
    """Compile the binding's extension module; its objects come from torch, already loaded when it is imported."""
    if not force and bind_fresh():
        return BIND
    import torch

    top = os.path.dirname(torch.__file__)
    tmp = BIND + ".%d.tmp" % os.getpid()
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", '-DVT_BIND_FOR="%s"' % bind_for(),
                           "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI, "-I", os.path.join(ROOT, "include"),
                           "-isystem", sysconfig.get_paths()["include"], "-isystem", os.path.join(top, "include"),
                           BIND_SRC, "-o", tmp, "-L", os.path.join(top, "lib"), "-lc10", "-ltorch_cpu", "-ltorch_python"])
    os.replace(tmp, BIND)
    return BIND


def build(force: bool = False, verbose: bool = False, stamps: bool = False) -> str:
    """Compile every .cu under csrc/ (one object each, in parallel) and link the shared library.
    stamps=True builds the instrumented twin (libvocabtrim_stamps.so, -DVT_STAMPS) instead."""
    LIB, OBJ_DIR = (LIB_STAMPS, OBJ_DIR_STAMPS) if stamps else (globals()["LIB"], globals()["OBJ_DIR"])
    build_bind(force)
    if not force and not needs_build(LIB):
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    os.makedirs(OBJ_DIR, exist_ok=True)
    extra = (["-Xptxas", "-v"] if verbose else []) + (["-DVT_STAMPS"] if stamps else [])
    procs, objs = [], []
    hdr_time = max(os.path.getmtime(p) for p in _deps() if not p.endswith(".cu"))
    for src in _sources():
        obj = os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if (not force and os.path.exists(obj) and os.path.getmtime(obj) > os.path.getmtime(src)
                and os.path.getmtime(obj) > hdr_time):
            continue
        cmd = [nvcc] + NVCC_FLAGS + extra + ["-c", src, "-o", obj]
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write("== %s\n%s\n" % (os.path.basename(src), out))
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB + ".%d.tmp" % os.getpid()
    subprocess.check_call([nvcc, "-shared", "-o", tmp] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv, stamps="--stamps" in sys.argv))
