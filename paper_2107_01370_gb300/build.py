"""In-tree build of liblbfsi.so (the C-ABI library) for sm_103a.

The translation units are compiled in parallel into objects under _build/
and linked into paper_2107_01370_gb300/liblbfsi.so.  No CMake, no torch
extension machinery: plain nvcc.
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
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(ROOT, "_build")
LIB = os.path.join(PKG, "liblbfsi.so")
# the bounds-checked variant (LBFSI_BOUNDS_CHECK: every shared-memory window
# and global slot of the step checked, a violation reported as LBFSI_EBOUNDS)
BUILD_BOUNDS = os.path.join(ROOT, "_build_bounds")
LIB_BOUNDS = os.path.join(PKG, "liblbfsi_bounds.so")
SOURCES = ["lbfsi_step.cu", "lbfsi_fields.cu", "lbfsi_stream64.cu", "lbfsi_elements.cu", "lbfsi_api.cu",
           "lbfsi_host.cu", "lbfsi_batch.cu", "lbfsi_noalloc.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2"]


# the step kernels' instantiations (tile shapes, launch forms) have to round
# alike: no contraction but the fused operations written out in their sources
SOURCE_FLAGS = {s: ["-fmad=false"] for s in ("lbfsi_step.cu", "lbfsi_fields.cu", "lbfsi_stream64.cu",
                                              "lbfsi_elements.cu")}


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _stale(target: str, deps: list[str]) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(verbose: bool = False, force: bool = False, bounds: bool = False) -> str:
    build_dir, lib = (BUILD_BOUNDS, LIB_BOUNDS) if bounds else (BUILD, LIB)
    extra = ["-DLBFSI_BOUNDS_CHECK"] if bounds else []
    os.makedirs(build_dir, exist_ok=True)
    headers = [os.path.join(CSRC, h) for h in os.listdir(CSRC) if h.endswith((".h", ".cuh"))]
    headers.append(os.path.join(INCLUDE, "lbfsi.h"))
    cc = nvcc()
    objs = []
    jobs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(build_dir, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + headers):
            jobs.append([cc, *ARCH, *FLAGS, *SOURCE_FLAGS.get(src, []), *extra, "-I", INCLUDE, "-I", CSRC, "-c", s, "-o", o])

    def run(cmd):
        if verbose:
            print(" ".join(cmd), flush=True)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed:\n{' '.join(cmd)}\n{r.stdout}\n{r.stderr}")
        return r

    with ThreadPoolExecutor(max_workers=len(jobs) or 1) as ex:
        list(ex.map(run, jobs))
    if force or jobs or _stale(lib, objs):
        run([cc, *ARCH, "-shared", "-o", lib, *objs, "-lcudart"])
    return lib


if __name__ == "__main__":
    print(build(verbose=True, force="--force" in sys.argv))
