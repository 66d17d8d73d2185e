"""Builds libmoe_b200.so (sm_100a only) and the binding's CPython helper in-tree.  `python -m paper_2606_26453_b200.build`."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
import warnings

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libmoe_b200.so")
# Test-only variant: device-side waits give up after 20 ms instead of 2 s, and a switch exists that withholds one
# barrier arrival so that a wait really runs out (tests/test_gpu_wait_timeout.py).  Never loaded by the binding.
WAITTEST_LIB_PATH = os.path.join(PKG_DIR, "libmoe_b200_waittest.so")
WAITTEST_FLAGS = ["-DMOE_TEST_HOOKS", "-DMOE_WAIT_LIMIT_NS=20000000ull"]
SOURCES = ["api.cu", "movement.cu", "router.cu", "grouped_gemm.cu", "mxfp8.cu"]
HEADERS = ["common.cuh", "tc_ptx.cuh", os.path.join("..", "..", "include", "moe_b200.h")]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def needs_build(path: str = LIB_PATH) -> bool:
    if not os.path.exists(path):
        return True
    t = os.path.getmtime(path)
    deps = [os.path.join(CSRC, s) for s in SOURCES + HEADERS]
    return any(os.path.getmtime(d) > t for d in deps)


PYCALL_PATH = os.path.join(PKG_DIR, "_pycall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
PYCALL_SOURCE = os.path.join(CSRC, "pycall.c")


def build_pycall(force: bool = False) -> str:
    """The module that marshals the binding's arguments (plain C, no CUDA)."""
    if force or not os.path.exists(PYCALL_PATH) or os.path.getmtime(PYCALL_SOURCE) > os.path.getmtime(PYCALL_PATH):
        cmd = [os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I" + sysconfig.get_path("include"), "-o", PYCALL_PATH, PYCALL_SOURCE]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError("gcc failed:\n" + res.stdout + res.stderr)
    return PYCALL_PATH


def build_library(force: bool = False, verbose: bool = False, waittest: bool = False) -> str:
    """The CUDA library, and the helper where it can be built (the binding does without it, with slower calls)."""
    path = WAITTEST_LIB_PATH if waittest else LIB_PATH
    if force or needs_build(path):
        _compile(path, verbose, waittest)
    try:
        build_pycall(force)
    except (OSError, RuntimeError) as e:
        warnings.warn(f"{os.path.basename(PYCALL_PATH)} was not built, calls of the binding will take longer: {e}", RuntimeWarning)
    return path


def _compile(path: str, verbose: bool, waittest: bool) -> None:
    cmd = [_nvcc(), "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
           "-shared", "-Xcompiler", "-fPIC", "-Xptxas", "-v" if verbose else "-warn-spills",
           "-o", path] + (WAITTEST_FLAGS if waittest else []) + [os.path.join(CSRC, s) for s in SOURCES]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    if verbose:
        print(res.stdout + res.stderr)


if __name__ == "__main__":
    print(build_library(force=True, verbose="-v" in sys.argv))
    print(build_library(force=True, waittest=True))
