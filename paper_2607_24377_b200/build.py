"""Build libmxattn.so in-tree with nvcc for sm_100a, and the CPython module that calls it (no JIT cache, no torch
extension machinery).

    python -m paper_2607_24377_b200.build          # rebuild if sources are newer than the library
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmxattn.so")
EXT = os.path.join(HERE, "_mxcall.so")          # CPython front end of the C ABI (csrc/pycall.cpp)
SOURCES = ["quantize.cu", "quantize_nvfp4.cu", "forward.cu", "forward_walk.cu", "forward_rows.cu", "forward_bf16.cu", "forward_nvfp4.cu", "rowsum_diag.cu", "fp4_gemm_probe.cu", "api.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC", "-shared",
]   # no fast-math: the quantizer relies on IEEE multiplies (subnormals are not flushed)


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def needs_build() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(EXT):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(EXT))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(HERE, "..", "include", "mxattn.h")]
    return any(os.path.getmtime(p) > t for p in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
          [os.path.join(CSRC, s) for s in SOURCES] + ["-o", LIB]
    ext = [shutil.which("g++") or "g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I" + sysconfig.get_paths()["include"],
           os.path.join(CSRC, "pycall.cpp"), "-o", EXT, "-L" + HERE, "-lmxattn", "-Wl,-rpath,$ORIGIN"]
    for what, c in (("libmxattn.so", cmd), ("_mxcall.so", ext)):
        res = subprocess.run(c, capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError("the compiler failed building " + what)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
