"""Builds the CUDA shared library in-tree (sm_100a only)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
ROOT = os.path.dirname(HERE)
LIB = os.path.join(HERE, "libsmartmem.so")
FASTCALL = os.path.join(HERE, "_fastcall" + sysconfig.get_config_var("EXT_SUFFIX"))   # CPython entry to the per-step calls (csrc/fastcall.c)

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC",
    "-cudart", "static",
]


def _sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cpp")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "smartmem.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build_fastcall() -> bool:
    """Compiles the CPython extension for the running interpreter.  It needs a C compiler and Python's headers; without them the per-step
    calls go through ctypes, about two microseconds of host time slower each."""
    cmd = [os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-Wall", "-I", sysconfig.get_paths()["include"], "-o", FASTCALL,
           os.path.join(CSRC, "fastcall.c")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write("the C compiler failed, the per-step calls go through ctypes:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
    return r.returncode == 0


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles every source under csrc/ into libsmartmem.so with nvcc; returns its path."""
    if not force and not _stale():
        if not os.path.exists(FASTCALL):                # (another interpreter's, perhaps)
            build_fastcall()
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, *NVCC_FLAGS, "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", LIB]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += _sources()
    cmd += ["-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
    build_fastcall()
    if verbose:
        sys.stderr.write(r.stderr)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
