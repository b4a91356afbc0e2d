"""Builds libss_msa.so (the C-ABI CUDA library, nvcc for sm_100a) and _pycall (the CPython side of the binding) in-tree."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
TRACE = bool(os.environ.get("SS_TRACE"))       # developer build with in-kernel timestamps
LIB = os.path.join(PKG, "libss_msa_trace.so" if TRACE else "libss_msa.so")
PYCALL = os.path.join(PKG, "_pycall" + sysconfig.get_config_var("EXT_SUFFIX"))
OBJ = os.path.join(PKG, "_build_trace" if TRACE else "_build")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC] + (["-DSS_TRACE"] if TRACE else [])
# Only the attention kernels are built with fast-math (ex2.approx, flush to zero).  Everything whose result is
# defined bit by bit (comparisons of logits, byte copies, single fp32 operations) keeps IEEE arithmetic.
FAST_MATH = {"ss_attention.cu"}


def nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: the CUDA library cannot be built")
    return exe


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every csrc/*.cu to an object and link them into libss_msa.so.  Incremental."""
    os.makedirs(OBJ, exist_ok=True)
    headers = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    objs, procs = [], []
    for src in sources():
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or _stale(obj, [src, *headers]):
            cmd = [nvcc(), *NVCC_FLAGS, *(["--use_fast_math"] if os.path.basename(src) in FAST_MATH else []), "-c", src, "-o", obj]
            if verbose:
                cmd.insert(1, "-Xptxas=-v")
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, pr in procs:
        out, _ = pr.communicate()
        if out.strip():
            print(out, file=sys.stderr)
        if pr.returncode != 0:
            failed = True
            print("nvcc failed on %s" % src, file=sys.stderr)
    if failed:
        raise RuntimeError("CUDA build failed")
    if procs or force or _stale(LIB, objs):
        tmp = LIB + ".tmp%d" % os.getpid()
        subprocess.check_call([nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp, *objs])
        os.replace(tmp, LIB)
    pycall = os.path.join(CSRC, "ss_pycall.cpp")
    if force or _stale(PYCALL, [pycall, os.path.join(ROOT, "include", "ss_msa.h")]):
        tmp = PYCALL + ".tmp%d" % os.getpid()
        subprocess.check_call([shutil.which("g++") or "g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", "-I",
                               os.path.join(ROOT, "include"), "-I", sysconfig.get_paths()["include"], pycall, "-o", tmp])
        os.replace(tmp, PYCALL)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
