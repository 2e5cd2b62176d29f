"""Build liblddmm.so in-tree with nvcc for sm_103a (GB300).

Compiles the CUDA translation units in parallel and links one shared
library with the CUDA runtime linked statically, so that loading it needs no
GPU.  Run ``python -m paper_1807_04638_gb300.build`` or call ``build()``.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OUT_DIR = os.path.join(HERE, "lib")
BUILD_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(OUT_DIR, "liblddmm.so")

# (source, object, defines): the passes are compiled once per number type, the
# stage kernels once per number type and last radix, the kernels of a compiled
# length once per length
SOURCES = [(f"{s}.cu", f"{s}_{t}.o", (f"-DLDDMM_T={t}",))
           for s in ("gen_pass", "fast_pass", "plane") for t in ("double", "float")]
SOURCES += [(f"{s}.cu", f"{s}.o", ()) for s in ("engine_f32", "engine_f64", "noalloc", "capi", "probe")]
SOURCES += [("stage_radix.cu", f"stage_{t}_{p}.o", (f"-DLDDMM_STAGE_T={t}", f"-DLDDMM_STAGE_P={p}"))
            for t, ps in (("float", (6, 5, 4, 3)), ("double", (10, 9, 8, 6, 5, 4))) for p in ps]
STAGE_LENGTHS = [384, 320, 300, 288, 270, 256, 250, 243, 240, 225, 216, 200, 192, 180, 162, 160, 150, 144, 135, 128, 125, 120, 108, 100, 96, 90, 81, 80, 75, 72, 64, 60, 54, 50, 48, 45, 40, 36, 32, 30, 27, 25, 24, 20, 18, 16]
SOURCES += [("stage_length.cu", f"stage_n{n}.o", (f"-DLDDMM_STAGE_N={n}",)) for n in STAGE_LENGTHS]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc_path() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build liblddmm.so")


def _flags(extra=()):
    return ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE,
                   "-I", CSRC, *extra]


def build(verbose: bool = False, extra_flags=()) -> str:
    """Compile and link; returns the path of the shared library."""
    nvcc = nvcc_path()
    os.makedirs(OUT_DIR, exist_ok=True)
    os.makedirs(BUILD_DIR, exist_ok=True)
    procs = []
    objs = []
    for src, name, defines in SOURCES:
        obj = os.path.join(BUILD_DIR, name)
        objs.append(obj)
        cmd = [nvcc, *_flags(extra_flags), *defines, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), flush=True)
        procs.append((name, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    failed = []
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(out.decode(errors="replace"))
        if p.returncode != 0:
            failed.append(src)
    if failed:
        raise RuntimeError(f"nvcc failed for {failed}")
    tmp = LIB + ".tmp"
    cmd = [nvcc, *ARCH, "-shared", "-cudart", "static", "-o", tmp, *objs]
    if verbose:
        print(" ".join(cmd), flush=True)
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv))
