"""Builds the CUDA library in-tree with nvcc for sm_100a, and the C extension through which Python makes its frequent calls
(no JIT cache, no fallback)."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libedgmoe.so")
CALLS = os.path.join(HERE, "_edgcall" + sysconfig.get_config_var("EXT_SUFFIX"))
CALLS_SRC = os.path.join(CSRC, "edg_python.c")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-shared", "-Xcompiler", "-fPIC",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h"))
    return any(os.path.getmtime(p) > t for p in deps)


def _run(cmd) -> str:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(os.path.basename(cmd[0]) + " failed:\n" + " ".join(cmd) + "\n" + res.stdout + res.stderr)
    return res.stderr


def build_calls(force: bool = False) -> str:
    """Compiles csrc/edg_python.c into _edgcall next to this file; returns its path."""
    deps = [CALLS_SRC] + glob.glob(os.path.join(INCLUDE, "*.h"))
    if force or not os.path.exists(CALLS) or any(os.path.getmtime(p) > os.path.getmtime(CALLS) for p in deps):
        _run([shutil.which("gcc") or shutil.which("cc") or "gcc", "-O2", "-std=gnu11", "-shared", "-fPIC", "-I", INCLUDE,
              "-I", sysconfig.get_path("include"), "-o", CALLS, CALLS_SRC])
    return CALLS


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles csrc/*.cu into libedgmoe.so next to this file; returns its path."""
    build_calls(force)
    if not force and not _stale():
        return LIB
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cmd = [nvcc, *NVCC_FLAGS, "-I", INCLUDE, "-o", LIB, *sources()]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    log = _run(cmd)
    if verbose:
        print(log)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
