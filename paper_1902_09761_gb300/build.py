"""Build libapfc.so (the CUDA library behind include/apfc.h) in-tree for sm_103a.

The translation units compile in parallel with nvcc, then link into
``paper_1902_09761_gb300/libapfc.so``.  Objects go to ``_build/``.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libapfc.so")
SOURCES = ["fused2d_v.cu", "fused2d_t.cu", "fused2d.cu", "kernels.cu", "stream3d.cu", "reduce.cu", "api.cu", "batch.cu", "noalloc.cu", "probe.cu", "resid2d.cu", "cheb2d_f32.cu", "cheb2d_f64.cu", "gauge2d_f32.cu", "gauge_tile.cu", "gauge_f64.cu", "resid_f64.cu", "schur.cu", "schur3d.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libapfc")
    return exe


def flags(extra=()):
    return [
        "-O3",
        "-lineinfo",
        "-std=c++17",
        *ARCH,
        "-Xcompiler",
        "-fPIC",
        "-I",
        os.path.join(ROOT, "include"),
        *extra,
    ]


def build(verbose: bool = False, extra_flags=()) -> str:
    os.makedirs(BUILD, exist_ok=True)
    exe = nvcc()
    procs = []
    objs = []
    for src in SOURCES:
        obj = os.path.join(BUILD, src.replace(".cu", ".o"))
        objs.append(obj)
        cmd = [exe, *flags(extra_flags), "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), flush=True)
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = []
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0:
            failed.append(f"--- {src}\n{out}")
        elif verbose and out.strip():
            print(out)
    if failed:
        raise RuntimeError("nvcc failed:\n" + "\n".join(failed))
    tmp = LIB + ".tmp"
    cmd = [exe, *ARCH, "-shared", *objs, "-o", tmp]
    r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n" + r.stdout)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv))
