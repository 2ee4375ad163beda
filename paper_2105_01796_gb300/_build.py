"""Build the CUDA library libkfgb.so in-tree (nvcc, sm_103a only)."""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libkfgb.so")
SOURCES = ["kf_kernels.cu", "kf_team.cu", "kf_mixed.cu", "kf_adjoint.cu", "kf_variants.cu", "kf_api.cu",
           "kf_static.cu"]
HEADERS = ["kf_internal.h", "kf_device.cuh", "kf_fp64.cuh", "kf_transport.cuh", "kf_team.cuh", "kf_filter.cuh", "kf_df.cuh",
           os.path.join("..", "..", "include", "kf.h")]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# per-file flags: the mixed kernel's FP32 divisions and square roots (step
# lengths, Jacobian normalisations, angle increments) need no IEEE rounding;
# its FP64 helpers use explicit intrinsics and are unaffected
# the warps of a track team each compute the state on their own and must take
# the same decisions, and the one-thread and the team kernels of the FP64 fit
# and of the adjoint give the same bits: their fused multiply-adds are written
# out, and the compiler contracts nothing more
FILE_FLAGS = {"kf_mixed.cu": ["-prec-div=false", "-prec-sqrt=false"],
              "kf_kernels.cu": ["-fmad=false"], "kf_team.cu": ["-fmad=false"], "kf_adjoint.cu": ["-fmad=false"]}


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libkfgb.so")


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + [os.path.join(CSRC, h) for h in HEADERS]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()
    flags = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2"]
    if verbose:
        flags += ["-Xptxas", "-v"]

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.splitext(src)[0] + ".o")
        cmd = [cc] + flags + FILE_FLAGS.get(src, []) + ["-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed for %s:\n%s" % (src, r.stderr))
        return obj, r.stderr

    with cf.ThreadPoolExecutor(len(SOURCES)) as ex:
        results = list(ex.map(compile_one, SOURCES))
    if verbose:
        for _, log in results:
            print(log)
    tmp = LIB + ".tmp"
    cmd = [cc] + ARCH + ["-shared", "-o", tmp] + [o for o, _ in results]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s" % r.stderr)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
