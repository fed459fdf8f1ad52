"""Build libdpsim.so in-tree with nvcc for sm_103a (GB300).

Translation units are compiled in parallel.  The physics and AMG-setup units
are compiled with -fmad=false so that their floating-point results are the
exact values of the formulas as written (no fused multiply-add); host code
is compiled with -ffp-contract=off for the same reason.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libdpsim.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
COMMON = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler",
          "-ffp-contract=off", "-I", os.path.join(ROOT, "include"), "-I", CSRC]
UNITS = {
    "dp_phys.cu": ["-fmad=false"],
    "dp_amg.cu": ["-fmad=false"],
    "dp_la.cu": [],
    "dp_sim.cu": [],
    "dp_noalloc.cu": [],
    "dp_cycle.cu": [],
    "dp_small.cu": [],
    "dp_serve.cu": [],
    "dp_batch.cu": [],
}


def _nvcc():
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if c and (os.path.sep not in c or os.path.exists(c)):
            return c
    return "nvcc"


def _stale(obj, deps):
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(BUILD, exist_ok=True)
    nvcc = _nvcc()
    headers = [os.path.join(CSRC, "dp_internal.h"), os.path.join(CSRC, "dp_kernels.cuh"),
               os.path.join(CSRC, "dp_tma.cuh"), os.path.join(CSRC, "dp_device.h"),
               os.path.join(CSRC, "dp_quotient.h"),
               os.path.join(ROOT, "include", "dpsim.h")]
    jobs = []
    objs = []
    for src, extra in UNITS.items():
        s = os.path.join(CSRC, src)
        o = os.path.join(BUILD, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s, __file__] + headers):
            jobs.append([nvcc, *ARCH, *COMMON, *extra, "-c", s, "-o", o])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        if verbose and (r.stdout or r.stderr):
            print(r.stdout + r.stderr)

    with cf.ThreadPoolExecutor(max_workers=len(UNITS)) as ex:
        list(ex.map(run, jobs))
    if force or jobs or _stale(LIB, objs):
        tmp = LIB + ".tmp"
        run([nvcc, *ARCH, "-shared", "-Xcompiler", "-fPIC", "-Xlinker", "-z,defs", *objs, "-ldl",
             "-o", tmp])
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose=True))
