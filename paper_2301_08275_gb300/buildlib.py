"""Build the CUDA library libgpe.so in-tree for sm_103a (nvcc, no cmake).

Each translation unit compiles in its own process (in parallel), then nvcc
links the shared library.  Rebuilds only when a source is newer than the
library.
"""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libgpe.so")
SOURCES = ["pass_f32_s1024_0.cu", "pass_f32_s1024_1.cu", "pass_f32_s512_0.cu", "pass_f32_s512_1.cu",
           "pass_f32_s256_0.cu", "pass_f32_s256_1.cu", "pass_f32_s64.cu", "pass_f32_s2048.cu",
           "pass_f32_r1024.cu", "pass_f32_r512.cu", "pass_f32_r256.cu", "pass_f32_r64.cu", "pass_f32_r2048.cu",
           "pass_f64_s1024.cu", "pass_f64_s512.cu", "pass_f64_s256.cu", "pass_f64_s128.cu", "pass_f64_s64.cu",
           "pass_f64_s2048.cu", "pass_f64_r1024.cu", "pass_f64_r512.cu", "pass_f64_r256.cu",
           "pass_f64_r128.cu", "pass_f64_r64.cu", "pass_f64_r2048.cu", "line1d_f64.cu", "line1d_f32.cu",
           "pass_f32.cu", "pass_f64.cu", "plane_cluster_f64.cu", "plane_cluster.cu", "diag_spec.cu", "api.cu",
           "noalloc.cu", "serve.cu", "peak.cu", "resident.cu", "line_cluster.cu"]
HEADERS = ["plane_cluster.cu", "fx.cuh", "fft_tile.cuh", "pass_kernels.cuh", "gpe_internal.h"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I" + os.path.join(ROOT, "include")]


def _nvcc():
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(BUILD, exist_ok=True)
    nvcc = _nvcc()
    hdrs = [os.path.join(CSRC, h) for h in HEADERS] + [os.path.join(ROOT, "include", h) for h in ("gpe.h", "gpe_serve.h")]
    objs, jobs = [], []
    for s in SOURCES:
        src = os.path.join(CSRC, s)
        obj = os.path.join(BUILD, s.replace(".cu", ".o"))
        objs.append(obj)
        if force or _stale(obj, [src] + hdrs):
            jobs.append([nvcc] + ARCH + FLAGS + ["-c", src, "-o", obj])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode:
            raise RuntimeError("nvcc failed: " + " ".join(cmd))

    if jobs:
        with ThreadPoolExecutor(max_workers=max(1, min(len(jobs), os.cpu_count() or 1))) as ex:
            list(ex.map(run, jobs))
    if force or jobs or _stale(LIB, objs):
        tmp = LIB + ".%d.tmp" % os.getpid()
        run([nvcc] + ARCH + ["-shared", "-o", tmp] + objs)
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
