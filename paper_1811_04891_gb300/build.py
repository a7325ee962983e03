"""Build the CUDA library libfindpts_gb.so in-tree for sm_103a (GB300).

Each translation unit is compiled by nvcc in parallel, then linked into one
shared library with the CUDA runtime linked statically.  Used by
``__graft_entry__.build()`` and on first import when the library is missing.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_build")
LIB = os.path.join(OUT, "libfindpts_gb.so")
SOURCES = ["fp_host.cu", "fp_setup.cu", "fp_scan.cu", "fp_find.cu", "fp_find2.cu", "fp_eval.cu", "fp_static.cu",
           "fp_batch.cu", "fp_flux.cu", "fp_stream.cu", "fp_probe.cu", "fp_solve.cu", "fp_tile_mixed.cu"]
HEADERS = ["fp_common.cuh", "fp_internal.h", "fp_handle.h", "fp_rank.cuh", "fp_newton.cuh", "fp_tile.cuh",
           "fp_tile_launch.cuh"]
# sources compiled once per order n, with flags of their own (the second's
# orders are those of is_tile_order in fp_internal.h; a missing one does not link)
PER_ORDER = {"fp_solve.cu": (range(2, 17), []), "fp_tile_mixed.cu": ([5, 7, 8, 9, 10], ["-fmad=false"])}
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _flags(extra=()):
    return ["-std=c++17", "-O3", "-lineinfo", *ARCH, "-Xcompiler", "-fPIC,-ffp-contract=off",
            "--expt-relaxed-constexpr", *extra]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(SRC, f) for f in SOURCES + HEADERS]
    deps.append(os.path.join(os.path.dirname(HERE), "include", "findpts_gb.h"))
    deps.append(os.path.abspath(__file__))
    return any(os.path.getmtime(d) > t for d in deps if os.path.exists(d))


def build(force: bool = False, verbose: bool = False, ptxas_v: bool = False) -> str:
    if not force and not _stale():
        return LIB
    os.makedirs(OUT, exist_ok=True)
    extra = ["-Xptxas", "-v"] if ptxas_v else []
    cmds, objs = [], []
    for f in SOURCES:
        orders, flags = PER_ORDER.get(f, ([0], []))
        for k in orders:
            objs.append(os.path.join(OUT, f.replace(".cu", f"_{k}.o" if k else ".o")))
            cmds.append([nvcc(), *_flags(extra), *flags, *([f"-DFP_N={k}"] if k else []), "-c", os.path.join(SRC, f),
                         "-o", objs[-1]])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        return cmd, r

    with cf.ThreadPoolExecutor(max_workers=len(cmds)) as ex:
        results = list(ex.map(run, cmds))
    for cmd, r in results:
        if verbose or ptxas_v:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed: " + " ".join(cmd) + "\n" + r.stdout + r.stderr)
    tmp = LIB + f".{os.getpid()}.tmp"
    link = [nvcc(), *ARCH, "-shared", "-o", tmp, *objs, "-Xcompiler", "-fPIC"]
    r = subprocess.run(link, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n" + r.stdout + r.stderr)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose=True, ptxas_v="-v" in sys.argv)
    print(LIB)
