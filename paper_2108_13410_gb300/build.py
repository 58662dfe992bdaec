"""Build the CUDA library libqsim.so in-tree (sm_103a only).

    python -m paper_2108_13410_gb300.build

One nvcc invocation per translation unit, in parallel, all for
-gencode arch=compute_103a,code=sm_103a, linked into
paper_2108_13410_gb300/_build/libqsim.so.
"""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OUT_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(OUT_DIR, "libqsim.so")
SOURCES = ["qsim.cu", "resident.cu", "noalloc.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _inputs():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files.append(os.path.join(INCLUDE, "qsim.h"))
    return files


def build(force: bool = False, verbose: bool = False, extra=None) -> str:
    os.makedirs(OUT_DIR, exist_ok=True)
    if not force and os.path.exists(LIB):
        t = os.path.getmtime(LIB)
        if all(os.path.getmtime(f) <= t for f in _inputs()):
            return LIB
    tmp = LIB + ".tmp%d" % os.getpid()
    cmd = [nvcc(), "-O3", "-std=c++17", *ARCH, "-lineinfo", "-Xcompiler", "-fPIC",
           "-I" + INCLUDE, "-I" + CSRC, "--expt-relaxed-constexpr"]
    if verbose:
        cmd.append("-Xptxas=-v")
    if extra:
        cmd += list(extra)

    def run(args):
        r = subprocess.run(args, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("nvcc failed building libqsim.so")
        if verbose:
            sys.stderr.write(r.stderr)

    objs = [os.path.join(OUT_DIR, "%s.%d.o" % (f, os.getpid())) for f in SOURCES]
    try:
        with ThreadPoolExecutor(len(SOURCES)) as ex:        # one nvcc per translation unit
            list(ex.map(run, [cmd + ["-c", os.path.join(CSRC, f), "-o", o] for f, o in zip(SOURCES, objs)]))
        run([nvcc(), *ARCH, "-shared", "-Xcompiler", "-fPIC", *objs, "-o", tmp, "-lcudart"])
    finally:
        for o in objs:
            if os.path.exists(o):
                os.remove(o)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
