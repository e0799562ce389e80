"""Compile the CUDA library in-tree with nvcc for sm_103a.

Each translation unit compiles to an object in parallel, then nvcc links them
into paper_1803_01756_gb300/_build/liblbm_gb300.so, a plain C ABI shared object
(include/lbm.h).  The units of the update kernels (PER_FILE) use approximate division and square
root (about 2 ulp) and flush denormals to zero (no value of the update comes within
30 orders of magnitude of the denormal range, so only the special-case code of
the reciprocal and root instructions goes away): instruction count bounds their
speed, and the results are checked against the FP64 oracle like every other path.
"""
from __future__ import annotations

import glob
import os
import subprocess
import threading
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "liblbm_gb300.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
COMMON = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC"]
_FAST = ["-prec-div=false", "-prec-sqrt=false", "-ftz=true"]
# The single-lattice fused kernel may take more registers for its schedule (156 instead of 150
# of the 168 that three CTAs per SM allow): GB300, 4096 x 512: 64.9 against 65.1 us per
# update, FP16 storage 70.5 against 71.2 us; 16384 x 2048: 902.5 against 904.7 us.
PER_FILE = {"lbm_fused.cu": _FAST + ["-Xptxas=--register-usage-level=8"]}
PER_FILE.update({f + ".cu": _FAST for f in (
    "lbm_fused_c2", "lbm_fused_batch", "lbm_twopass", "lbm_sweep", "lbm_sweep_f16",
    "lbm_sweep_bf16", "lbm_sweep_batch", "lbm_sweep_batch_f16", "lbm_sweep_batch_bf16", "lbm_tile", "lbm_tile_f16", "lbm_tile_bf16")})
_lock = threading.Lock()


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _inputs():
    return sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(
        os.path.join(CSRC, "*.h")) + [os.path.join(ROOT, "include", "lbm.h"), __file__]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _compile(src: str, verbose: bool) -> str:
    obj = os.path.join(BUILD, os.path.basename(src) + f".{os.getpid()}.o")
    cmd = [nvcc(), *ARCH, *COMMON, *PER_FILE.get(os.path.basename(src), []),
           "-I", os.path.join(ROOT, "include"), "-c", src, "-o", obj]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    subprocess.run(cmd, check=True)
    return obj


def build(force: bool = False, verbose: bool = False) -> str:
    with _lock:
        newest = max(os.path.getmtime(p) for p in _inputs())
        if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= newest:
            return LIB
        os.makedirs(BUILD, exist_ok=True)
        srcs = sources()
        with ThreadPoolExecutor(max_workers=len(srcs)) as ex:
            objs = list(ex.map(lambda s: _compile(s, verbose), srcs))
        tmp = LIB + f".{os.getpid()}.tmp"
        try:
            subprocess.run([nvcc(), *ARCH, "-shared", "-o", tmp, *objs], check=True)
        finally:
            for o in objs:
                if os.path.exists(o):
                    os.remove(o)
        os.replace(tmp, LIB)
        return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
