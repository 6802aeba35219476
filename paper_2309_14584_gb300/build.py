"""Build the in-tree CUDA library libfct_gb300.so for sm_103a with nvcc.

The translation units (host tables, the library's host code and small
kernels, and three per block size for the team solver kernels) are compiled in
parallel and linked into one shared library (static CUDA runtime), next to
this file.  No torch headers are used:
the library's ABI is plain C (include/fct.h).
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libfct_gb300.so")

SOURCES = ["fct_solve_k256.cu", "fct_solve_k128.cu", "fct_solve_k512.cu", "fct_solve_k256d.cu", "fct_solve_k128d.cu",
           "fct_solve_k512d.cu", "fct_solve_k256c.cu", "fct_solve_k128c.cu", "fct_solve_k512c.cu", "fct_device.cu",
           "fct_plan_device.cu", "fct_plan_host.cpp", "fct_peaks.cu", "fct_dct_tc.cu"]
HEADERS = ["fct_internal.h", "fct_df.cuh", "fct_common.cuh", "fct_solver.cuh", "fct_cells.cuh"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libfct_gb300.so")


def _inputs():
    files = [os.path.join(CSRC, s) for s in SOURCES]
    files += [os.path.join(CSRC, h) for h in HEADERS] + [os.path.join(INCLUDE, "fct.h"), __file__]
    return files


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(f) <= t for f in _inputs())


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False) -> str:
    if not force and up_to_date():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()
    # template kernel stubs get external linkage, so that host code in one
    # translation unit can launch the solver kernels instantiated in another
    # host code rounds every floating-point operation on its own (no fused
    # multiply-add), so host- and device-built tables agree bit for bit on
    # x86 and Arm hosts alike
    common = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-ffp-contract=off",
                     "-static-global-template-stub=false", "-I", INCLUDE, "-I", CSRC]
    if ptxas_info:
        common += ["-Xptxas", "-v"]
    procs, objs = [], []
    for src in SOURCES:
        obj = os.path.join(BUILD, os.path.splitext(src)[0] + ".o")
        cmd = [cc] + common + ["-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        procs.append((cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    for cmd, p in procs:
        out, _ = p.communicate()
        if verbose or ptxas_info:
            sys.stderr.write(out)
        if p.returncode != 0:
            raise RuntimeError(f"nvcc failed ({p.returncode}): {' '.join(cmd)}\n{out}")
    tmp = LIB + ".tmp"
    link = [cc] + ARCH + ["-shared", "-o", tmp] + objs
    r = subprocess.run(link, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed: {' '.join(link)}\n{r.stdout}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv))
