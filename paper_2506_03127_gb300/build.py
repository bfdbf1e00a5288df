"""Build libqp.so in-tree with nvcc for sm_103a (GB300).

    python -m paper_2506_03127_gb300.build

The translation units (qp.cu in seven parts, mlp.cu, wide.cu, host_numerics.cpp) are compiled in parallel, then linked into
paper_2506_03127_gb300/libqp.so.  A rebuild happens only when a source is
newer than the library (or force=True).
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libqp.so")
BUILD = os.path.join(PKG, "_build")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
SOURCES = ["qp.cu", "mlp.cu", "wide.cu", "host_numerics.cpp"]
# qp.cu is compiled once per unit: its tile kernels are spread over units 1 .. 6
JOBS = [("qp.cu", u) for u in range(7)] + [(s, None) for s in SOURCES[1:]]
HEADERS = ["internal.h"]


def _nvcc():
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found; the CUDA toolkit is required to build libqp")
    return cand


def _stale(force: bool) -> bool:
    if force or not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES + HEADERS] + [os.path.join(ROOT, "include", "qp.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False) -> str:
    if not _stale(force):
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    nvcc = _nvcc()
    common = ["-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include")]

    def compile_one(job):
        src, unit = job
        obj = os.path.join(BUILD, src + (".o" if unit is None else f".{unit}.o"))
        cmd = [nvcc, "-c", os.path.join(CSRC, src), "-o", obj] + common
        if unit is not None:
            cmd += [f"-DQP_UNIT={unit}"]
        if src.endswith(".cu"):
            cmd += ARCH + ["-lineinfo"]
            if ptxas_info:
                cmd += ["-Xptxas", "-v"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        if verbose and (r.stdout or r.stderr):
            print(r.stdout + r.stderr, file=sys.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=len(JOBS)) as ex:
        objs = list(ex.map(compile_one, JOBS))
    tmp = LIB + ".tmp"
    cmd = [nvcc, "-shared", "-o", tmp] + objs + ARCH + ["-lcudart_static", "-lrt", "-lpthread", "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_info="-v" in sys.argv))
