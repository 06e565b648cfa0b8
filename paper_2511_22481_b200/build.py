"""Builds the C-ABI shared library (libomni_mla.so) in-tree with nvcc for sm_100a, and the CPython
module that binding.py calls it through (_marshal) with g++ against PyTorch's headers."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libomni_mla.so")
SOURCES = [os.path.join(CSRC, "api.cu"), os.path.join(CSRC, "static_scratch.cu")]
MARSHAL = os.path.join(HERE, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))
MARSHAL_SOURCE = os.path.join(CSRC, "marshal.cpp")


def _deps():
    out = [os.path.join(ROOT, "include", "omni_mla.h")]
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            out.append(os.path.join(CSRC, name))
    return out


def needs_build() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(p) > t for p in _deps())


def build_marshal(force: bool = False) -> str:
    """Compile the CPython module; it finds libomni_mla.so next to itself and PyTorch's libraries in the
    process that imports it."""
    deps = (MARSHAL_SOURCE, os.path.join(ROOT, "include", "omni_mla.h"))
    if not force and os.path.exists(MARSHAL) and all(os.path.getmtime(p) <= os.path.getmtime(MARSHAL) for p in deps):
        return MARSHAL
    from torch.utils import cpp_extension
    tmp = MARSHAL + ".tmp.%d" % os.getpid()
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-I", os.path.join(ROOT, "include"),
           "-I", os.path.join(cuda, "include"), "-I", sysconfig.get_paths()["include"]]
    for path in cpp_extension.include_paths():
        cmd += ["-isystem", path]
    cmd += [MARSHAL_SOURCE, "-o", tmp, LIB, "-Wl,-rpath,$ORIGIN"]
    for path in cpp_extension.library_paths():
        cmd += ["-L", path]
    cmd += ["-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("g++ failed building _marshal")
    os.replace(tmp, MARSHAL)
    return MARSHAL


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile the library (every CUDA source) and the CPython module; returns the library's path."""
    if not force and not needs_build():
        build_marshal()
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "--shared", "-Xcompiler", "-fPIC", "-Xlinker", "-soname=libomni_mla.so", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", tmp] + SOURCES
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed building libomni_mla.so")
    os.replace(tmp, LIB)
    build_marshal(force)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
