"""Builds libtgp.so (host planner + engine + sm_100a kernels) in-tree with nvcc, and the extension that calls it from Python without ctypes."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libtgp.so")
FASTCALL = os.path.join(HERE, "_fastcall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
SOURCES = ["tgp_host.cpp", "tgp_model.cpp", "tgp_kernels.cu", "tgp_gemm_sm100.cu", "tgp_attn_prefill.cu", "tgp_attn_sm100.cu", "tgp_engine.cu"]


def sources():
    return [os.path.join(CSRC, s) for s in SOURCES if os.path.exists(os.path.join(CSRC, s))] + \
           [os.path.join(CSRC, f) for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cpp")) and f not in SOURCES]


def needs_build() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(FASTCALL):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(FASTCALL))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
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
    cmd = [os.environ.get("CC", "gcc"), "-O2", "-Wall", "-fPIC", "-shared", "-I" + INCLUDE, "-I" + sysconfig.get_paths()["include"], "-o", FASTCALL, os.path.join(CSRC, "tgp_fastcall.c")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("the Python extension does not build:\n" + r.stdout + r.stderr)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
