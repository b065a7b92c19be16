"""Builds the CUDA library in-tree with nvcc for sm_100a, and the extension module that calls it.

    python -m paper_2307_14995_b200.build [--force] [--verbose]

Produces ``paper_2307_14995_b200/libla_b200.so`` (C ABI declared in
``include/la.h``) and the extension module ``_la_call``, whose file name carries the tag of the interpreter that it was
built for, so that no other one loads it.  Needs nvcc (which cross-compiles without a GPU), a C compiler ($CC, or gcc) and
Python's headers.
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libla_b200.so")
CALL = os.path.join(HERE, "_la_call" + sysconfig.get_config_var("EXT_SUFFIX"))
UNTAGGED_CALL = os.path.join(HERE, "_la_call.so")  # as it was once built: any interpreter would load it
SOURCES = ["la_api.cu", "la_simt.cu", "la_decode.cu", "la_tc.cu", "la_noalloc.cu", "la_gate.cu", "la_lrpe.cu"]
HEADERS = ["la_common.cuh", os.path.join("..", "..", "include", "la.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps if os.path.exists(d))


def build(force: bool = False, verbose: bool = False) -> str:
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    hdrs = [os.path.join(CSRC, h) for h in HEADERS] + [
        os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    objs = []
    procs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(objdir, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + hdrs):
            cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", s, "-o", o]
            procs.append((cmd, subprocess.Popen(cmd)))
    for cmd, p in procs:
        if p.wait() != 0:
            raise RuntimeError("nvcc failed: " + " ".join(cmd))
    if force or procs or _stale(LIB, objs):
        tmp = LIB + ".tmp%d" % os.getpid()
        cmd = [_nvcc(), "-shared", "-o", tmp] + objs + ["-lcudart"]
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    src = os.path.join(CSRC, "la_call.c")
    if force or _stale(CALL, [src]):
        tmp = CALL + ".tmp%d" % os.getpid()
        subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC", "-I" + sysconfig.get_paths()["include"],
                               src, "-o", tmp])
        os.replace(tmp, CALL)
    if os.path.exists(UNTAGGED_CALL):
        os.remove(UNTAGGED_CALL)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
