"""Compile the CUDA library in-tree with nvcc for sm_100a (one object per source file, then one shared library)."""
from __future__ import annotations

import glob
import os
import re
import shutil
import subprocess
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
OBJ = os.path.join(CSRC, "build")
LIB = os.path.join(_HERE, "libzipline.so")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC"]


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def headers() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h"))
                  + glob.glob(os.path.join(INCLUDE, "*.h")))


def _changed(src: str) -> float:
    """When the source, or a source that it includes, was last changed."""
    included = re.findall(r'^#include "(\w+\.cu)"', open(src).read(), re.M)
    return max(os.path.getmtime(f) for f in [src] + [os.path.join(CSRC, i) for i in included])


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the ZipLine CUDA library cannot be built")


def _obj(src: str) -> str:
    return os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(d) > t for d in sources() + headers())


def build(force: bool = False, verbose: bool = False) -> str:
    """Build ``libzipline.so`` next to this file when missing or older than its sources."""
    if not (force or is_stale()):
        return LIB
    nvcc = _nvcc()
    os.makedirs(OBJ, exist_ok=True)
    newest_header = max(os.path.getmtime(h) for h in headers())
    todo = [s for s in sources()
            if force or not os.path.exists(_obj(s)) or os.path.getmtime(_obj(s)) < max(_changed(s), newest_header)]

    def compile_one(src: str):
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", "-o", _obj(src), src]
        return subprocess.run(cmd, cwd=CSRC, capture_output=True, text=True)

    with ThreadPoolExecutor(max(1, min(len(todo), 4, os.cpu_count() or 1))) as ex:
        results = list(ex.map(compile_one, todo))
    for src, r in zip(todo, results):
        if verbose or r.returncode != 0:
            print(f"--- {os.path.basename(src)}\n{r.stdout}{r.stderr}", flush=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.run([nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp] + [_obj(s) for s in sources()],
                   check=True, cwd=CSRC)
    os.replace(tmp, LIB)
    return LIB
