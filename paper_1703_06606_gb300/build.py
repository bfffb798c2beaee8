"""Build the CUDA libraries in-tree for sm_103a (GB300).

    python -m paper_1703_06606_gb300.build [--force] [--verbose]

Translation units are compiled in parallel with one -gencode
(arch=compute_103a, code=sm_103a) and linked into
paper_1703_06606_gb300/libqnsch.so (the solver's C ABI, include/qnsch.h) and
paper_1703_06606_gb300/libqnsch_probe.so (the FMA throughput and issue-cost
probes that measure the FP64 roofline's denominator; measurement tooling, not
part of the solver's ABI), both next to this file.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(ROOT, "_build")
LIB = os.path.join(HERE, "libqnsch.so")
PROBE_LIB = os.path.join(HERE, "libqnsch_probe.so")
SOURCES = ["kernels.cu", "solver.cu", "noalloc.cu"]
PROBE_SOURCES = ["probe.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# the host passes stop at an object read as one of another class: the optimiser
# may assume that no such read happens
HOST = ["-Xcompiler", "-fPIC,-Werror=strict-aliasing,-Wstrict-aliasing=1"]


def nvcc():
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _deps():
    out = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    out.append(os.path.join(INCLUDE, "qnsch.h"))
    return out


def is_stale():
    for lib in (LIB, PROBE_LIB):
        if not os.path.exists(lib):
            return True
        t = os.path.getmtime(lib)
        if any(os.path.getmtime(d) > t for d in _deps()):
            return True
    return False


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not is_stale():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    flags = ARCH + HOST + ["-O3", "-lineinfo", "-std=c++17", "-I", INCLUDE, "-I", CSRC]
    if verbose:
        flags += ["-Xptxas", "-v"]

    def compile_one(src):
        obj = os.path.join(BUILD, src.replace(".cu", ".o"))
        cmd = [nvcc()] + flags + ["-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed on %s:\n%s\n%s" % (src, r.stdout, r.stderr))
        return obj, r.stderr

    with cf.ThreadPoolExecutor(len(SOURCES) + len(PROBE_SOURCES)) as ex:
        res = list(ex.map(compile_one, SOURCES + PROBE_SOURCES))
    if verbose:
        for _, err in res:
            sys.stderr.write(err)
    objs = [o for o, _ in res]
    for lib, part in ((LIB, objs[:len(SOURCES)]), (PROBE_LIB, objs[len(SOURCES):])):
        tmp = lib + ".tmp%d" % os.getpid()
        cmd = [nvcc()] + ARCH + ["-shared", "-o", tmp] + part
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("link failed:\n%s\n%s" % (r.stdout, r.stderr))
        os.replace(tmp, lib)
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="--verbose" in sys.argv)
    print(LIB)
