"""Build the CUDA library in-tree: ``python -m paper_2210_00129_b200.build``.

Compiles every ``csrc/*.cu`` for sm_100a with nvcc into ``libsbp_b200.so`` next to this file, and
``csrc/python_calls.cpp`` into the CPython module of the calls where Python's headers are installed
(the binding goes through ctypes otherwise).  Cross-compiles without a GPU.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB_PATH = os.path.join(_HERE, "libsbp_b200.so")

CALLS_SRC = os.path.join(CSRC, "python_calls.cpp")
CALLS_PATH = os.path.join(_HERE, "_calls" + sysconfig.get_config_var("EXT_SUFFIX"))

NVCC_FLAGS = ["-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
              "-Xcompiler", "-fPIC", "-shared"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _has_python_headers() -> bool:
    return os.path.exists(os.path.join(sysconfig.get_paths()["include"], "Python.h"))


def _stale(out: str, deps) -> bool:
    return not os.path.exists(out) or any(os.path.getmtime(d) > os.path.getmtime(out) for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    header = os.path.join(os.path.dirname(_HERE), "include", "sbp.h")
    jobs = [(LIB_PATH, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + [header],
             [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB_PATH] + sources())]
    if _has_python_headers():
        jobs.append((CALLS_PATH, [CALLS_SRC, header],
                     [nvcc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-cudart", "none", "-I", sysconfig.get_paths()["include"],
                      "-o", CALLS_PATH, CALLS_SRC, "-L", _HERE, "-Xlinker", "-l:" + os.path.basename(LIB_PATH), "-Xlinker", "-rpath,$ORIGIN"]))
    for out, deps, cmd in jobs:
        if not force and not _stale(out, deps):
            continue
        res = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError("nvcc failed building " + os.path.basename(out))
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
