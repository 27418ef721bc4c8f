"""Builds liblumo_gdn.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a.

    python -m paper_2609_23900_b200.build [--force] [--verbose]

nvcc cross-compiles without a GPU.  The shared object is placed next to this file so
that it travels with the source tree; what ptxas says of each kernel (registers, spills)
is kept beside the object files, in build/<source>.ptxas.
"""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liblumo_gdn.so")
SOURCES = ["api.cu", "kernels.cu", "scan_gram.cu", "scan_solve.cu", "scan_stream.cu", "attn.cu", "kv_cache.cu", "accept.cu", "select.cu", "tree_desc.cpp"]
HEADERS = [os.path.join(CSRC, "internal.h"), os.path.join(CSRC, "call_order.h"), os.path.join(CSRC, "conv_split.h"), os.path.join(ROOT, "include", "lumo_gdn.h")]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + HEADERS + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not (force or _stale()):
        return LIB
    objs = []
    os.makedirs(os.path.join(HERE, "build"), exist_ok=True)
    for src in SOURCES:
        obj = os.path.join(HERE, "build", src + ".o")
        cmd = [_nvcc(), *NVCC_FLAGS, "-Xptxas", "-v", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-x", "cu",
               "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), flush=True)
        done = subprocess.run(cmd, stderr=subprocess.PIPE, text=True)
        if verbose or done.returncode:
            print(done.stderr, file=sys.stderr, flush=True)
        done.check_returncode()
        with open(os.path.join(HERE, "build", src + ".ptxas"), "w") as f:
            f.write(done.stderr)
        objs.append(obj)
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.check_call([_nvcc(), "-shared", "-gencode", "arch=compute_100a,code=sm_100a", *objs, "-o", tmp])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
