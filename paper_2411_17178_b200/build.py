"""Builds liblitevar.so (the C-ABI library, nvcc, sm_100a) and _litevar_host.*.so (its Python entry, C compiler) in-tree.

    python -m paper_2411_17178_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liblitevar.so")
HOST_LIB = os.path.join(HERE, "_litevar_host" + sysconfig.get_config_var("EXT_SUFFIX"))  # of this interpreter
HOST_SOURCE = os.path.join(CSRC, "litevar_host.c")
SOURCES = ["litevar_plan.cu", "litevar_fwd_simt.cu", "litevar_maps.cu", "litevar_fwd_ws.cu", "litevar_fwd_small.cu", "litevar_static.cu", "litevar_calib.cu", "litevar_quant.cu"]
HEADERS = [os.path.join(CSRC, "litevar_internal.h"), os.path.join(CSRC, "litevar_tc_ptx.h"), os.path.join(ROOT, "include", "litevar.h")]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _stale(target: str, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def needs_build() -> bool:
    return _stale(LIB, [os.path.join(CSRC, s) for s in SOURCES] + HEADERS + [os.path.abspath(__file__)])


def build_host(force: bool = False) -> str:
    if force or _stale(HOST_LIB, [HOST_SOURCE, HEADERS[-1], os.path.abspath(__file__)]):
        cmd = [os.environ.get("CC") or "gcc", "-shared", "-fPIC", "-O2", "-Wall", "-I", sysconfig.get_paths()["include"],
               "-I", os.path.join(ROOT, "include"), HOST_SOURCE, "-o", HOST_LIB]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError("building _litevar_host.so failed:\n" + res.stdout + res.stderr)
    return HOST_LIB


def build(force: bool = False, verbose: bool = False) -> str:
    build_host(force)
    if not force and not needs_build():
        return LIB
    cmd = [_nvcc(), "-shared", "-Xcompiler", "-fPIC", "-O3", "-std=c++17", "-lineinfo",
           "-gencode", "arch=compute_100a,code=sm_100a",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "--cudart", "shared"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", LIB]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed building liblitevar.so")
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
