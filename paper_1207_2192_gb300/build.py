"""Build libnanodisk.so (the C-ABI library) in-tree with nvcc for sm_103a.

The translation units are compiled in parallel and linked into
``paper_1207_2192_gb300/_build/libnanodisk.so``.  Runs on x86_64 (cross
compile, no GPU needed) and on the aarch64 GPU hosts alike.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "libnanodisk.so")
SOURCES = ["nd_fused_f32.cu", "nd_fused_f64.cu", "nd_cluster_f32.cu", "nd_cluster_f64.cu", "nd_glob_f32.cu", "nd_glob_f64.cu",
           "nd_dispatch.cu", "nd_aux.cu", "nd_api.cu", "nd_noalloc.cu", "nd_spectra.cu",
           "nd_energy.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# The stepping, relaxation and field kernels write their fused multiply-adds
# out (fm in nd_common.cuh): without contraction by the compiler every
# schedule of a step rounds alike, whichever kernel it is inlined into.
NO_CONTRACT = {"nd_fused_f32.cu", "nd_fused_f64.cu", "nd_cluster_f32.cu", "nd_cluster_f64.cu", "nd_glob_f32.cu", "nd_glob_f64.cu", "nd_noalloc.cu"}


def nvcc() -> str:
    for c in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found")


def _flags(verbose_ptxas: bool = False):
    f = ARCH + ["-O3", "-lineinfo", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC",
                "-Xcompiler", "-O2", "-Xcompiler", "-ffp-contract=off"]
    if verbose_ptxas:
        f += ["-Xptxas", "-v"]
    return f


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(HERE, "..", "include", "nanodisk.h"), __file__]
    return any(os.path.getmtime(d) > t for d in deps if os.path.exists(d))


def build(force: bool = False, verbose_ptxas: bool = False, jobs: int | None = None) -> str:
    """Compile (if stale) and return the path of libnanodisk.so."""
    if not force and not _stale():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()
    objs = []

    def one(src):
        obj = os.path.join(BUILD, src.replace(".cu", ".o"))
        exact = ["-fmad=false"] if src in NO_CONTRACT else []
        cmd = [cc] + _flags(verbose_ptxas) + exact + ["-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stderr}")
        return obj, r.stderr

    with cf.ThreadPoolExecutor(max_workers=jobs or len(SOURCES)) as ex:
        results = list(ex.map(one, SOURCES))
    logs = []
    for obj, err in results:
        objs.append(obj)
        logs.append(err)
    tmp = LIB + ".tmp"
    r = subprocess.run([cc] + ARCH + ["-shared", "-o", tmp] + objs, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stderr}")
    os.replace(tmp, LIB)
    if verbose_ptxas:
        with open(os.path.join(BUILD, "ptxas.log"), "w") as f:
            f.write("\n".join(logs))
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose_ptxas="-v" in sys.argv))
