"""Builds the in-tree CUDA library ``libswf.so`` for sm_103a (GB300) with nvcc.

Each translation unit compiles in parallel; the objects link into one shared library next to
this file.  Nothing is installed outside the repository.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libswf.so")
SOURCES = ["swf_api.cu", "swf_march.cu", "swf_project.cu", "swf_fused.cu", "swf_noalloc.cu", "swf_bw.cu", "swf_mlp.cu",
           "swf_pairs.cu"]
# the register line kernels: one unit per list of lengths (swf_line_list.h)
LINE_LISTS = 5
UNITS = [(src, [], os.path.splitext(src)[0]) for src in SOURCES] + [
    ("swf_line.cu", [f"-DSWF_LINE_LIST={i}", "-DSWF_LINE_REAL=float"], f"swf_line{i}") for i in range(LINE_LISTS)]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


def nvcc() -> str:
    path = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(path):
        raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libswf.so")
    return path


def _compile(unit, verbose: bool) -> str:
    src, defines, name = unit
    obj = os.path.join(OUT_DIR, name + ".o")
    cmd = [nvcc(), *ARCH, *FLAGS, *defines, "-c", os.path.join(CSRC, src), "-o", obj]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{res.stdout}\n{res.stderr}")
    if verbose and res.stderr:
        sys.stderr.write(res.stderr)
    return obj


def build(verbose: bool = False, force: bool = False) -> str:
    """Compile every CUDA source into libswf.so (skipped when the library is newer)."""
    os.makedirs(OUT_DIR, exist_ok=True)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps.append(os.path.join(HERE, "..", "include", "swf.h"))
    if not force and os.path.exists(LIB):
        lib_t = os.path.getmtime(LIB)
        if all(os.path.getmtime(d) <= lib_t for d in deps):
            return LIB
    with ThreadPoolExecutor(max_workers=max(4, os.cpu_count() or 4)) as ex:
        objs = list(ex.map(lambda u: _compile(u, verbose), UNITS))
    tmp = LIB + ".tmp"
    cmd = [nvcc(), *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link failed:\n{res.stdout}\n{res.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, force="-f" in sys.argv))
