"""Builds libtgp.so (host planner + engine + sm_100a kernels) in-tree with nvcc, and the extension that calls it from Python without ctypes."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libtgp.so")
FASTCALL = os.path.join(HERE, "_fastcall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
SOURCES = ["tgp_host.cpp", "tgp_model.cpp", "tgp_kernels.cu", "tgp_gemm_sm100.cu", "tgp_attn_prefill.cu", "tgp_attn_sm100.cu", "tgp_engine.cu"]


def sources():
    return [os.path.join(CSRC, s) for s in SOURCES if os.path.exists(os.path.join(CSRC, s))] + \
           [os.path.join(CSRC, f) for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cpp")) and f not in SOURCES]


def _stale(target, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def _lib_stale() -> bool:
    return _stale(LIB, [os.path.join(d, f) for d in (CSRC, INCLUDE) for f in os.listdir(d) if f != "tgp_fastcall.c"])


def _fastcall_stale() -> bool:
    return _stale(FASTCALL, [os.path.join(CSRC, "tgp_fastcall.c")] + [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)])


def needs_build() -> bool:
    return _lib_stale() or _fastcall_stale()


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _lib_stale():
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
               "-Xcompiler", "-fPIC", "-shared", "-I" + INCLUDE, "-I" + CSRC, "-o", LIB] + sources()
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + r.stdout + r.stderr)
        if verbose:
            sys.stderr.write(r.stderr)
    if force or _fastcall_stale():
        _build_fastcall()
    return LIB


def _build_fastcall() -> None:
    """The extension takes host time off calls that ctypes serves as well, so a machine without a C compiler or Python's headers gets a warning.  What an
    earlier build left goes: it may not be the library's any more."""
    cmd = [os.environ.get("CC", "gcc"), "-O2", "-Wall", "-fPIC", "-shared", "-I" + INCLUDE, "-I" + sysconfig.get_paths()["include"], "-o", FASTCALL, os.path.join(CSRC, "tgp_fastcall.c")]
    try:
        r = subprocess.run(cmd, capture_output=True, text=True)
        why = f"{cmd[0]} ended with {r.returncode}\n{r.stdout}{r.stderr}" if r.returncode else None
    except OSError as e:
        why = str(e)
    if why:
        if os.path.exists(FASTCALL):
            os.remove(FASTCALL)
        warnings.warn("the Python extension does not build, its calls go through ctypes:\n" + why, RuntimeWarning)


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
