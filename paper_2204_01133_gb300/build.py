"""Compile the CUDA library libat_gb300.so in-tree (nvcc, sm_103a only).

Usage: ``python -m paper_2204_01133_gb300.build`` (or ``build()``).  Each
translation unit is compiled in parallel, then linked into a shared library
with the CUDA runtime linked statically, so the library depends only on the
driver.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "libat_gb300.so")
PROBE = os.path.join(HERE, "libat_probe.so")
BUILD = os.path.join(HERE, "_build")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# one object each; the step-fused kernels by halo width (the longest to compile)
SOURCES = ["at_fused.cu:-DAT_FUSED_H=1", "at_fused.cu:-DAT_FUSED_H=2", "at_fused.cu:-DAT_FUSED_H=3", "at_fused.cu",
           "at_stage.cu", "at_abi.cu", "at_persist.cu", "at_cluster.cu", "at_tilefused.cu"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "--fmad=true", "-Xptxas", "-O3"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is needed to build libat_gb300.so")


def _stale() -> bool:
    if not os.path.exists(OUT) or not os.path.exists(PROBE):
        return True
    t = os.path.getmtime(OUT)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps.append(os.path.join(HERE, "..", "include", "at.h"))
    deps.append(os.path.abspath(__file__))
    return any(os.path.getmtime(d) > t for d in deps if os.path.exists(d))


def build(force: bool = False, verbose: bool = False, extra=()) -> str:
    if not force and not _stale():
        return OUT
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()

    def compile_one(unit):
        src, *defs = unit.split(":")
        obj = os.path.join(BUILD, src.replace(".cu", "") + "".join(d[-1] for d in defs) + ".o")
        cmd = [cc, *ARCH, *FLAGS, *extra, *defs, "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed on %s:\n%s%s" % (src, r.stdout, r.stderr))
        if verbose:
            sys.stdout.write(r.stdout + r.stderr)
        return obj

    with ThreadPoolExecutor(len(SOURCES) + 1) as ex:
        objs = list(ex.map(compile_one, SOURCES + ["fp64_probe.cu"]))
    probe_obj = objs.pop()
    r = subprocess.run([cc, *ARCH, "-shared", "-o", PROBE + ".tmp", probe_obj, "-cudart", "static"],
                       capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("probe link failed:\n%s%s" % (r.stdout, r.stderr))
    os.replace(PROBE + ".tmp", PROBE)
    tmp = OUT + ".tmp"
    cmd = [cc, *ARCH, "-shared", "-o", tmp, *objs, "-cudart", "static"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s%s" % (r.stdout, r.stderr))
    os.replace(tmp, OUT)
    return OUT


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv,
                extra=["-Xptxas", "-v"] if "-v" in sys.argv else ()))
