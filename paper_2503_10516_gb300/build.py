"""Builds libigs.so (the C-ABI library) for sm_103a with nvcc, in-tree.

Each object file is compiled in parallel, then all are linked into
``_build/libigs.so``. The lowering engine is inlined into each of its
kernels and takes most of the time, so they are objects of their own (one
source). The executor's TU is built with ``-fmad=false`` so the float workload
kernels round after every operation.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "libigs.so")
INCLUDE = os.path.join(ROOT, "include")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# object file: source and its own flags
OBJECTS = {
    **{f"igs_lower{k}.o": ("igs_lower.cu", [f"-DIGS_LOWER_PART={k}"]) for k in range(5)},
    "igs_exec.o": ("igs_exec.cu", ["-fmad=false"]),
    "igs_host.o": ("igs_host.cu", []),
    "igs_static.o": ("igs_static.cu", []),
}


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _deps_mtime() -> float:
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, "igs.h")]
    return max(os.path.getmtime(f) for f in files)


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    os.makedirs(BUILD, exist_ok=True)
    if (not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _deps_mtime() and not extra_flags
            and not os.environ.get("IGS_PROFILE_DETAIL")):
        return LIB
    nvcc = _nvcc()
    common = ["-std=c++17", "-O3", "-lineinfo", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC] + ARCH + list(extra_flags)
    if os.environ.get("IGS_PROFILE_DETAIL"):
        common.append("-DIGS_PROFILE_DETAIL")

    def compile_one(name):
        src, flags = OBJECTS[name]
        obj = os.path.join(BUILD, name)
        cmd = [nvcc, "-c", os.path.join(CSRC, src), "-o", obj] + common + flags
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {name}:\n{r.stderr}")
        if verbose and r.stderr:
            sys.stderr.write(r.stderr)
        return obj

    with cf.ThreadPoolExecutor(max_workers=len(OBJECTS)) as ex:
        objs = list(ex.map(compile_one, OBJECTS))
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [nvcc, "-shared", "-o", tmp] + objs + ARCH + ["-lcudart"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv,
                extra_flags=["-Xptxas", "-v"] if "--ptxas" in sys.argv else ()))
