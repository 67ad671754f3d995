"""Builds the CUDA library (``libdion_b200.so``) in-tree with nvcc for sm_100a.

Run as ``python -m paper_2504_05295_b200.build`` (``-f`` compiles everything, ``-v`` does and shows
ptxas's report) or through ``__graft_entry__.build()``.  nvcc cross-compiles, so no GPU is needed.
The translation units are compiled side by side; an object is reused while none of the files it
includes is newer.
"""
from __future__ import annotations

import os
import re
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdion_b200.so")
OBJ_DIR = os.path.join(HERE, "_obj")
SOURCES = ["dion_api.cu", "umma_gemm.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


def _includes(path: str, seen: set) -> set:
    """`path` and every file of this repository that it includes."""
    if path in seen:
        return seen
    seen.add(path)
    with open(path) as f:
        for name in re.findall(r'^\s*#include\s+"([^"]+)"', f.read(), re.M):
            for folder in (CSRC, os.path.join(ROOT, "include")):
                if os.path.exists(os.path.join(folder, name)):
                    _includes(os.path.join(folder, name), seen)
    return seen


def _newest(source: str) -> float:
    return max(os.path.getmtime(p) for p in _includes(os.path.join(CSRC, source), set()))


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= max(_newest(s) for s in SOURCES):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ_DIR, exist_ok=True)
    running, objects = [], []
    for s in SOURCES:
        obj = os.path.join(OBJ_DIR, os.path.splitext(s)[0] + ".o")
        objects.append(obj)
        if not force and os.path.exists(obj) and os.path.getmtime(obj) >= _newest(s):
            continue
        tmp = f"{obj}.tmp{os.getpid()}"
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else [])
        cmd += ["-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", os.path.join(CSRC, s), "-o", tmp]
        running.append((subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True), tmp, obj))
    failed = ""
    for proc, tmp, obj in running:
        out = proc.communicate()[0]
        if verbose:
            sys.stderr.write(out)
        if proc.returncode != 0:
            failed += out
        else:
            os.replace(tmp, obj)
    if failed:
        raise RuntimeError("nvcc failed:\n" + failed)
    tmp = LIB + f".tmp{os.getpid()}"
    res = subprocess.run([nvcc] + NVCC_FLAGS[:2] + ["-shared", "-Xcompiler", "-fPIC"] + objects + ["-o", tmp, "-lcudart"],
                         capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed to link:\n" + res.stdout + res.stderr)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="-f" in sys.argv or "-v" in sys.argv, verbose="-v" in sys.argv))
