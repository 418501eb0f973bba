"""Compile the CUDA library in-tree: paper_2601_16986_b200/libcrystalkv.so (sm_100a only)."""
from __future__ import annotations

import glob
import os
import subprocess
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcrystalkv.so")
HEADER = os.path.join(os.path.dirname(HERE), "include", "crystalkv.h")


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")) + [HEADER])


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and os.path.exists(LIB):
        if all(os.path.getmtime(LIB) >= os.path.getmtime(s) for s in _sources()):
            return LIB
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    flags = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC"]
    if verbose:
        flags.append("-Xptxas=-v")
    with tempfile.TemporaryDirectory() as tmp:   # one compiler per unit, side by side
        objs = [os.path.join(tmp, os.path.basename(s) + ".o") for s in srcs]
        procs = [subprocess.Popen(["nvcc", *flags, "-c", "-o", o, s]) for s, o in zip(srcs, objs)]
        failed = [s for p, s in zip(procs, srcs) if p.wait() != 0]
        if failed:
            raise RuntimeError(f"nvcc failed on {failed}")
        subprocess.run(["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", LIB + ".tmp", *objs], check=True)
    os.replace(LIB + ".tmp", LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
