"""Build libtaot.so (sm_100a only) in-tree with nvcc.  `python -m paper_2608_03676_b200.build`."""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libtaot.so")
OBJ = os.path.join(PKG, "csrc", "build")
SOURCES = ["api.cu", "histogram.cu", "sinkhorn.cu", "sinkhorn_cluster.cu", "sinkhorn_dense_tc.cu", "sinkhorn_class.cu", "sinkhorn_wide.cu", "sinkhorn_tiered.cu", "sinkhorn_tile.cu", "sinkhorn_tile_r32.cu", "sinkhorn_tile_r32_batch.cu", "sinkhorn_tile_r64.cu", "sinkhorn_tile_r64_batch.cu", "sinkhorn_tile_r256_batch.cu", "match.cu", "assign.cu", "report.cu", "peaks.cu", "dispatch.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xptxas", "-v",
              "-I", os.path.join(ROOT, "include"), "-I", CSRC] + os.environ.get("TAOT_EXTRA_NVCC_FLAGS", "").split()


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    headers = [os.path.join(CSRC, "taot_internal.cuh"), os.path.join(CSRC, "sinkhorn_common.cuh"), os.path.join(CSRC, "sinkhorn_generic.cuh"),
               os.path.join(CSRC, "sinkhorn_tile.cuh"), os.path.join(CSRC, "sinkhorn_split.cuh"), os.path.join(CSRC, "sinkhorn_class.h"), os.path.join(CSRC, "auction.cuh"),
               os.path.join(ROOT, "include", "taot.h"), os.path.join(ROOT, "include", "taot_measure.h")]
    nvcc = _nvcc()

    def compile_one(src: str):
        s = os.path.join(CSRC, src)
        o = os.path.join(OBJ, src.replace(".cu", ".o"))
        if force or _stale(o, [s] + headers):
            r = subprocess.run([nvcc] + NVCC_FLAGS + ["-c", s, "-o", o], capture_output=True, text=True)
            with open(o + ".log", "w") as f:
                f.write(r.stdout + r.stderr)
            if r.returncode != 0:
                raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
            if verbose:
                print(r.stderr)
        return o

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    if force or _stale(LIB, objs):
        r = subprocess.run([nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB] + objs,
                           capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
