"""Builds libflowblock.so (sm_100a) in-tree with nvcc, and the binding's
marshalling module (csrc/marshal.c) with the C compiler.

``python -m paper_2607_17652_b200.build`` or :func:`build`.  Cross-compiles
without a GPU.  Objects are rebuilt only when a source or header is newer.
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
ROOT = os.path.dirname(HERE)
LIB = os.path.join(HERE, "libflowblock.so")
# named for the Python it is built against: another one does not load it
MARSHAL = os.path.join(HERE, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))
SOURCES = ["api.cu", "pack.cu", "t2t.cu", "gate_commit.cu", "attn_sm100.cu", "scatter.cu", "lm_head.cu",
           "attn_static.cu", "attn_pair_sm100.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo",
              "-std=c++17", "-Xcompiler", "-fPIC", "-Xptxas", "-v"]


def _nvcc() -> str:
    cand = os.environ.get("NVCC") or os.path.join(
        os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _deps():
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    hs.append(os.path.join(ROOT, "include", "flowblock.h"))
    return hs


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(os.path.join(HERE, "build"), exist_ok=True)
    hdr_time = max(os.path.getmtime(h) for h in _deps())
    jobs = []
    objs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(HERE, "build", src.replace(".cu", ".o"))
        objs.append(o)
        if force or not os.path.exists(o) or \
                os.path.getmtime(o) < max(os.path.getmtime(s), hdr_time):
            jobs.append([_nvcc(), *NVCC_FLAGS, "-c", s, "-o", o])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode:
            sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        if r.returncode:
            raise RuntimeError("the compiler failed for " + cmd[-3])
        return r.stderr

    with ThreadPoolExecutor(max_workers=4) as ex:
        logs = list(ex.map(run, jobs))
    if jobs or not os.path.exists(LIB) or force:
        run([_nvcc(), "-shared", "-o", LIB, *objs, "-gencode",
             "arch=compute_100a,code=sm_100a"])
    untagged = os.path.join(HERE, "_marshal.so")        # what earlier builds left, which any Python would load
    if os.path.exists(untagged):
        os.remove(untagged)
    src = os.path.join(CSRC, "marshal.c")
    if force or not os.path.exists(MARSHAL) or \
            os.path.getmtime(MARSHAL) < max(os.path.getmtime(src), hdr_time):
        run([os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-Wall",
             "-I", sysconfig.get_paths()["include"], src, "-o", MARSHAL])
    if logs:
        with open(os.path.join(HERE, "build", "ptxas.log"), "w") as f:
            f.write("\n".join(logs))
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
