"""Builds the C-ABI shared library in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB_PATH = os.path.join(HERE, "libtorq_b200.so")
SOURCES = [os.path.join(CSRC, "torq.cu")]
BINDING_PATH = os.path.join(HERE, "_torq_binding" + sysconfig.get_config_var("EXT_SUFFIX"))
BINDING_SOURCE = os.path.join(CSRC, "binding.cpp")


def _deps():
    out = [os.path.join(HERE, "..", "include", "torq.h")]
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh", ".h")):
            out.append(os.path.join(CSRC, f))
    return out


def needs_build() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    return any(os.path.getmtime(p) > t for p in _deps())


def needs_binding() -> bool:
    if not os.path.exists(BINDING_PATH):
        return True
    t = os.path.getmtime(BINDING_PATH)
    return any(os.path.getmtime(p) > t for p in (BINDING_SOURCE, os.path.join(HERE, "..", "include", "torq.h")))


def build_binding(force: bool = False) -> str:
    """The native marshalling of the layer calls (a CPython extension; it reads tensors through torch's headers)."""
    if not force and not needs_binding():
        return BINDING_PATH
    from torch.utils import cpp_extension
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-o", BINDING_PATH, BINDING_SOURCE,
           "-I" + sysconfig.get_paths()["include"], "-I/usr/local/cuda/include"]
    cmd += ["-I" + p for p in cpp_extension.include_paths()]
    for p in cpp_extension.library_paths():
        cmd += ["-L" + p]
    cmd += ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("g++ failed: " + " ".join(cmd))
    return BINDING_PATH


def build_library(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared", "-o", LIB_PATH] + SOURCES
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed: " + " ".join(cmd))
    return LIB_PATH


if __name__ == "__main__":
    print(build_library(force=True, verbose="-v" in sys.argv))
    print(build_binding(force=True))
