"""Build libpgb.so in-tree (paper_1506_03745_gb300/_build/) with nvcc for sm_103a.

Every translation unit is compiled in parallel, then linked into one shared
library with the CUDA runtime linked statically.  Run as
``python -m paper_1506_03745_gb300.build``.
"""
import concurrent.futures
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_build")
LIB = os.path.join(OUT, "libpgb.so")
SOURCES = ["tree.cu", "matvec.cu", "treecode_f32.cu", "treecode_f64.cu", "solver.cu", "energy.cu", "adjoint.cu",
           "imposed_f32.cu", "treecode_ds.cu", "treecode_ds_hi.cu", "batch.cu", "farfield.cu", "shard.cu", "api.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# --no-compress: nvcc compresses device code beyond some size, and its first kernel in a process then waits for
# the expansion (7 ms for the FP64 treecode's)
FLAGS = ["-O3", "--no-compress", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-pthread", "-Xcompiler", "-Wno-deprecated-declarations"]


def nvcc():
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found")
    return exe


def _stale(obj, deps):
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    return any(os.path.getmtime(d) > t for d in deps)


def build(verbose=False, force=False):
    os.makedirs(OUT, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(os.path.dirname(HERE), "include", "pgb.h"))
    exe = nvcc()
    jobs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(OUT, src.replace(".cu", ".o"))
        if force or _stale(o, [s] + headers):
            jobs.append([exe] + ARCH + FLAGS + ["-c", s, "-o", o])
    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        return cmd[-1]
    with concurrent.futures.ThreadPoolExecutor(max_workers=max(1, min(len(jobs), os.cpu_count() or 4))) as ex:
        for o in ex.map(run, jobs):
            if verbose:
                print("compiled", o)
    objs = [os.path.join(OUT, s.replace(".cu", ".o")) for s in SOURCES]
    if force or jobs or not os.path.exists(LIB):
        tmp = LIB + ".tmp"
        run([exe] + ARCH + ["-shared", "-o", tmp] + objs)
        os.replace(tmp, LIB)
        if verbose:
            print("linked", LIB)
    return LIB


if __name__ == "__main__":
    build(verbose=True, force="--force" in sys.argv)
