"""In-tree build of the CUDA library ``libbidiag.so`` for sm_103a (nvcc + g++, no cmake).

``python -m paper_1611_06892_gb300.build`` or ``build()``: compiles the translation units in parallel
into ``paper_1611_06892_gb300/_build/`` and links ``paper_1611_06892_gb300/libbidiag.so``.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libbidiag.so")
ROOT = os.path.dirname(HERE)

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# (source, value of BD_EXEC_PART): kernels.cu is compiled once per executor instantiation; diagnostic 177 (unused
# function) is off because each of these compilations uses only a part of the file
UNITS = [("kernels.cu", part) for part in (1, 2, 3, 4, 5, 0)] + [
    (src, None) for src in ("plan.cpp", "capi.cu", "noalloc.cu", "peak.cu")]


def _nvcc():
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libbidiag.so")
    return cand


def _compile(unit, verbose):
    src, part = unit
    nvcc = _nvcc()
    obj = os.path.join(BUILD, os.path.splitext(src)[0] + ("" if part is None else f"_{part}") + ".o")
    cmd = [nvcc, "-std=c++17", "-O3", "-lineinfo", "-Xcompiler", "-fPIC,-O2", "-diag-suppress", "177", *ARCH,
           "-I", os.path.join(ROOT, "include"), "-c", os.path.join(CSRC, src), "-o", obj]
    cmd += [] if part is None else [f"-DBD_EXEC_PART={part}"]
    if src.endswith(".cu"):
        cmd += ["-Xptxas", "-v"] if verbose else []
    else:
        cmd += ["-x", "c++"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"compile of {src} failed:\n{' '.join(cmd)}\n{res.stdout}\n{res.stderr}")
    return obj, res.stderr


def build(verbose=False):
    os.makedirs(BUILD, exist_ok=True)
    with ThreadPoolExecutor(max_workers=len(UNITS)) as ex:
        outs = list(ex.map(lambda u: _compile(u, verbose), UNITS))
    if verbose:
        for _, log in outs:
            if log:
                print(log, file=sys.stderr)
    tmp = LIB + ".tmp"
    cmd = [_nvcc(), "-shared", *ARCH, "-o", tmp, *[o for o, _ in outs], "-lcudart", "-lpthread"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link failed:\n{' '.join(cmd)}\n{res.stdout}\n{res.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv))
