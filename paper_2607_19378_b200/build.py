"""Builds libhyenand.so in-tree with nvcc for sm_100a (no JIT cache involved).

    python -m paper_2607_19378_b200.build [--force] [--verbose] [--debug] [--lineinfo]
"""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "build")
LIB = os.path.join(HERE, "libhyenand.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "--use_fast_math", "-Xptxas", "-v"]
# A kernel's first launch in a process loads its source file's whole device image.  The product library therefore holds it as it
# is, without line tables, which are two thirds of it (65 MB in all).  First forward of a process, against one stored compressed
# for size with line tables (36 MB): 262144-point lines 17.7 -> 4.1 ms, 512x512 planes 29.3 -> 7.3, 64x64 planes 9.8 -> 1.8.  The
# checked build has both, line tables and compression; --lineinfo gives the product library its line tables for a profiler.
PRODUCT_FLAGS = ["--compress-mode=none"]
DEBUG_FLAGS = ["-lineinfo", "--compress-mode=size", "-DHYENAND_DEBUG"]
# --use_fast_math: approximate division and exponentials, subnormals flushed.  The transforms themselves use neither (their
# twiddles come from tables computed in double on the host).  What does are the gates and norms of Eq. 2 (mixer.cu, and
# mix_sigmoid inside fused2d.cu and slice_mix*.cu), at fp32 errors of a few 1e-7; 1 / (1 + exp(x)) is 0 above x = 87.3, where
# it is below 2^-126.  Kernel synthesis, whose sines reach 30 radians and more, is compiled without it.
PRECISE = {"synth.cu"}


def _sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _newest_header():
    t = 0.0
    for root in (CSRC, os.path.join(os.path.dirname(HERE), "include")):
        for f in os.listdir(root):
            if f.endswith((".cuh", ".h")):
                t = max(t, os.path.getmtime(os.path.join(root, f)))
    return t


def build(force: bool = False, verbose: bool = False, debug: bool = False, lineinfo: bool = False) -> str:
    """Compiles and links the library; debug=True builds the checked variant (-DHYENAND_DEBUG) as libhyenand_debug.so."""
    OBJ = os.path.join(HERE, "build_debug" if debug else "build")
    LIB = os.path.join(HERE, "libhyenand_debug.so" if debug else "libhyenand.so")
    os.makedirs(OBJ, exist_ok=True)
    hdr = _newest_header()
    extra = DEBUG_FLAGS if debug else PRODUCT_FLAGS + (["-lineinfo"] if lineinfo else [])
    jobs = []
    objs = []
    for src in _sources():
        s = os.path.join(CSRC, src)
        o = os.path.join(OBJ, src[:-3] + ".o")
        objs.append(o)
        if force or not os.path.exists(o) or os.path.getmtime(o) < max(os.path.getmtime(s), hdr):
            jobs.append((s, o))

    def compile_one(job):
        s, o = job
        flags = [f for f in FLAGS if not (f == "--use_fast_math" and os.path.basename(s) in PRECISE)] + extra
        r = subprocess.run([NVCC] + flags + ["-c", s, "-o", o], capture_output=True, text=True)
        with open(o[:-2] + ".ptxas.log", "w") as f:
            f.write(r.stderr)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {s}:\n{r.stderr[-4000:]}")
        if verbose:
            print(r.stderr)
        return o

    if jobs:
        with ThreadPoolExecutor(max_workers=min(8, len(jobs))) as ex:
            list(ex.map(compile_one, jobs))
    stale = not os.path.exists(LIB) or any(os.path.getmtime(o) > os.path.getmtime(LIB) for o in objs)
    manifest = os.path.join(OBJ, "objects.txt")
    listed = open(manifest).read() if os.path.exists(manifest) else ""
    if jobs or stale or listed != "\n".join(objs):
        tmp = LIB + ".tmp.%d" % os.getpid()
        subprocess.check_call([NVCC, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp] + objs + ["-lcudart", "-ldl"])
        os.replace(tmp, LIB)
        with open(manifest, "w") as f:
            f.write("\n".join(objs))
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv, debug="--debug" in sys.argv,
                lineinfo="--lineinfo" in sys.argv))
