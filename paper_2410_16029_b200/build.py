"""Compile the C-ABI library in-tree with nvcc for sm_100a, and the Python binding's helper with the host compiler.

``python -m paper_2410_16029_b200.build`` (or ``build_library()``) writes
``libngalore.so`` and ``_bind.so`` next to this file.  nvcc cross-compiles without a GPU.
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "csrc", "ngalore_api.cu")
OUT = os.path.join(HERE, "libngalore.so")
BIND_SRC = os.path.join(HERE, "csrc", "bind.cpp")
BIND_OUT = os.path.join(HERE, "_bind.so")
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC", "-cudart", "static"]


def _sources():
    d = os.path.join(HERE, "csrc")
    inc = os.path.join(os.path.dirname(HERE), "include", "ngalore.h")
    return [os.path.join(d, f) for f in os.listdir(d) if f.endswith((".cu", ".cuh"))] + [inc]


def _bind_stamp() -> str:
    """What _bind.so depends on beside its source."""
    import torch

    return "torch %s, Python %s" % (torch.__version__, ".".join(map(str, sys.version_info[:3])))


def _bind_current(out: str, stamp: str) -> bool:
    """Whether `out` is newer than its source and was built with what `stamp` says."""
    try:
        with open(out + ".stamp") as f:
            return f.read() == stamp and os.path.getmtime(out) >= os.path.getmtime(BIND_SRC)
    except OSError:
        return False


def _build_bind(force: bool) -> None:
    stamp = _bind_stamp()
    if not force and _bind_current(BIND_OUT, stamp):
        return
    import torch

    home = os.path.dirname(torch.__file__)
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + sysconfig.get_paths()["include"],
           "-I" + os.path.join(home, "include"), "-I" + os.path.join(home, "include", "torch", "csrc", "api", "include"),
           "-o", BIND_OUT, BIND_SRC, "-L" + os.path.join(home, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("host compiler failed: " + " ".join(cmd))
    with open(BIND_OUT + ".stamp", "w") as f:
        f.write(stamp)


def build_library(force: bool = False, verbose: bool = False) -> str:
    _build_bind(force)
    if not force and os.path.exists(OUT):
        newest = max(os.path.getmtime(p) for p in _sources())
        if os.path.getmtime(OUT) >= newest:
            return OUT
    nvcc = os.environ.get("NVCC", "nvcc")
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", OUT, SRC]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("nvcc failed: " + " ".join(cmd))
    if verbose:
        sys.stderr.write(res.stderr)
    return OUT


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
