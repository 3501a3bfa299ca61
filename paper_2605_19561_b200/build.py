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


def binding_path() -> str:
    """The binding is compiled against torch's C++ headers, so a file serves one torch version: it carries that in its name."""
    import torch
    return os.path.join(HERE, "_torq_binding-torch" + torch.__version__ + sysconfig.get_config_var("EXT_SUFFIX"))


def needs_binding() -> bool:
    path = binding_path()
    if not os.path.exists(path):
        return True
    t = os.path.getmtime(path)
    return any(os.path.getmtime(p) > t for p in (BINDING_SOURCE, os.path.join(HERE, "..", "include", "torq.h")))


def _compile(cmd, path, verbose=False):
    """Runs `cmd` + [-o <file beside path>] and moves the result to `path` in one step: processes that start together and find
    it missing each build their own, and none loads a file that another is still writing."""
    tmp = os.path.join(os.path.dirname(path), f".{os.getpid()}.{os.path.basename(path)}")
    try:
        res = subprocess.run(cmd + ["-o", tmp], capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError(os.path.basename(cmd[0]) + " failed: " + " ".join(cmd))
        os.replace(tmp, path)
    finally:
        if os.path.exists(tmp):
            os.remove(tmp)
    return path


def build_binding(force: bool = False) -> str:
    """The native marshalling of the layer calls (a CPython extension; it reads tensors through torch's headers)."""
    path = binding_path()
    if not force and not needs_binding():
        return path
    from torch.utils import cpp_extension
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", BINDING_SOURCE, "-I" + sysconfig.get_paths()["include"]]
    cmd += ["-I" + p for p in cpp_extension.include_paths("cuda")]
    cmd += ["-L" + p for p in cpp_extension.library_paths()]
    return _compile(cmd + ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python"], path)


def build_library(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared"] + SOURCES
    if verbose:
        cmd[1:1] = ["-Xptxas", "-v"]
    return _compile(cmd, LIB_PATH, verbose)


if __name__ == "__main__":
    print(build_library(force=True, verbose="-v" in sys.argv))
    print(build_binding(force=True))
