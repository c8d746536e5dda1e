"""Builds librmsmp.so (the C-ABI CUDA library, nvcc for sm_100a) and the extension module that marshals its per-layer
calls, both in-tree."""
from __future__ import annotations

import os
import shutil
import subprocess
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "librmsmp.so")
MARSHAL_SOURCE = os.path.join(CSRC, "marshal.cpp")
# named for the interpreter it was built for, so that another one does not load it
MARSHAL = os.path.join(_HERE, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))
SOURCES = ("host_api.cu", "pack.cu", "simt.cu", "tensor.cu", "tensor2.cu", "split.cu", "peak.cu", "builtin_scratch.cu", "stream.cu", "assign.cu", "depthwise.cu", "gather.cu")
HEADERS = tuple(sorted(f for f in os.listdir(CSRC) if f.endswith((".cuh", ".h")))) + \
          (os.path.join("..", "..", "include", "rmsmp.h"),)

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--fmad=false",                       # quantizer arithmetic is one IEEE operation per step
    "-Xcompiler", "-fPIC,-ffp-contract=off,-O2",
    "-shared",
    "-ldl",                               # the NVTX header loads a profiler's library on demand
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA library cannot be built")


def _older(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps if os.path.exists(d))


def needs_build() -> bool:
    return _older(LIB, [os.path.join(CSRC, s) for s in SOURCES + HEADERS] + [os.path.abspath(__file__)])


def build_marshal(force: bool = False) -> str:
    """The CPython extension (host code only: no CUDA headers, nothing linked)."""
    header = os.path.join(CSRC, "..", "..", "include", "rmsmp.h")
    if not force and not _older(MARSHAL, [MARSHAL_SOURCE, header, os.path.abspath(__file__)]):
        return MARSHAL
    untagged = os.path.join(_HERE, "_marshal.so")         # the name of earlier builds, which any interpreter would load
    if os.path.exists(untagged):
        os.remove(untagged)
    tmp = MARSHAL + ".%d.tmp" % os.getpid()
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], MARSHAL_SOURCE, "-o", tmp])
    os.replace(tmp, MARSHAL)
    return MARSHAL


def build_library(force: bool = False, verbose: bool = False) -> str:
    build_marshal(force)
    if not force and not needs_build():
        return LIB
    tmp = LIB + ".%d.tmp" % os.getpid()
    cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
          [os.path.join(CSRC, s) for s in SOURCES] + ["-o", tmp]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build_library(force=True, verbose="-v" in sys.argv))
