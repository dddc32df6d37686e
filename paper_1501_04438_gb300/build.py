"""Build libgsm.so in this directory with nvcc for sm_103a (GB300).

    python -m paper_1501_04438_gb300.build [--force]

Translation units compile in parallel; the result is linked into a shared
library with a C ABI (include/gsm.h) and the CUDA runtime linked statically.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libgsm.so")
# the units that take longest to compile first
SOURCES = [*(f"gsm_fx_split_{u}.cu" for u in "abcde"), *(f"gsm_fx_len_{u}.cu" for u in "abcdefghijkl"), "gsm_passes.cu",
           "gsm_fx_queue3d.cu", "gsm_fx_queue2d.cu", "gsm_fx3_c.cu", "gsm_fx3_a.cu", "gsm_fx3_b.cu", "gsm_f3_f32.cu",
           "gsm_fx.cu", "gsm_fx_conv.cu", "gsm_conv_rr.cu", "gsm_tc.cu", "gsm_plan.cu", "gsm_api.cu"]
HEADERS = ["gsm_arith.cuh", "gsm_fft.cuh", "gsm_fx.cuh", "gsm_fx_passes.cuh", "gsm_fx_kernels.cuh", "gsm_fx_split.cuh",
           "gsm_fx3.cuh", "gsm_f3_f32.cuh", "gsm_fx_queue.cuh", "gsm_pass_common.cuh", "gsm_internal.h"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "--compress-mode=size", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(BUILD, exist_ok=True)
    hdrs = [os.path.join(CSRC, h) for h in HEADERS] + [os.path.join(HERE, "..", "include", "gsm.h")]
    objs, jobs = [], []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(BUILD, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + hdrs):
            jobs.append([nvcc(), *ARCH, *FLAGS, "-c", s, "-o", o])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        if verbose and (r.stdout or r.stderr):
            print(r.stdout + r.stderr, file=sys.stderr)

    with cf.ThreadPoolExecutor(max_workers=max(1, len(jobs))) as ex:
        list(ex.map(run, jobs))
    if force or jobs or _stale(LIB, objs):
        tmp = LIB + ".tmp"
        run([nvcc(), *ARCH, "-shared", "-cudart", "static", *objs, "-o", tmp])
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
