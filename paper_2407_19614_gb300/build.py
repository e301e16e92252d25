"""Build librihf.so (CUDA, sm_103a) in-tree with nvcc; no cmake, no torch extension.

    python -m paper_2407_19614_gb300.build [--debug]

Each translation unit is compiled in parallel; the shared library lands next to
this file as ``librihf.so`` and object files under ``_build/``.
"""

from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "librihf.so")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
SOURCES = ["rihf_api.cu", "grad_eri3_lane.cu", "grad_one_lane.cu", "eri3_lane.cu", "one_lane.cu", "eri2_lane.cu", "integrals.cu", "grad_integrals.cu", "linalg.cu", "eigh_tridiag.cu", "jk.cu", "eigh_noalloc.cu", "tc_gemm.cu", "mlp.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc():
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _compile(src, debug):
    obj = os.path.join(OUT, os.path.splitext(os.path.basename(src))[0] + ".o")
    flags = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", SRC,
             "--expt-relaxed-constexpr", "-rdc=false"]
    if debug:
        flags += ["-DRIHF_DEBUG"]
    cmd = [nvcc(), *ARCH, *flags, "-c", os.path.join(SRC, src), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, r.stdout, r.stderr))
    return obj, r.stderr


def build(debug: bool = False, verbose: bool = False) -> str:
    os.makedirs(OUT, exist_ok=True)
    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        results = list(ex.map(lambda s: _compile(s, debug), SOURCES))
    objs = [o for o, _ in results]
    if verbose:
        for _, err in results:
            if err.strip():
                print(err, file=sys.stderr)
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc(), *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s\n%s" % (r.stdout, r.stderr))
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(debug="--debug" in sys.argv, verbose=True))
