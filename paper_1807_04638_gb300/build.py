"""Build liblddmm.so in-tree with nvcc for sm_103a (GB300).

Compiles the CUDA translation units in parallel and links one shared
library with the CUDA runtime linked statically, so that loading it needs no
GPU.  Run ``python -m paper_1807_04638_gb300.build`` or call ``build()``.
"""
from __future__ import annotations

import os
import re
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OUT_DIR = os.path.join(HERE, "lib")
BUILD_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(OUT_DIR, "liblddmm.so")


def stage_lengths():
    """The compiled line lengths, longest first: LDDMM_STAGE_LENGTHS of stage.cuh."""
    with open(os.path.join(CSRC, "stage.cuh")) as f:
        table = re.search(r"#define LDDMM_STAGE_LENGTHS\(X\)((?:.*\\\n)*.*\n)", f.read()).group(1)
    return sorted((int(n) for n in re.findall(r"X\((\d+),", table)), reverse=True)


# (source, object, defines): the passes are compiled once per number type, the
# stage kernels once per number type and last radix, the kernels of a compiled
# length once per length
SOURCES = [(f"{s}.cu", f"{s}_{t}.o", (f"-DLDDMM_T={t}",))
           for s in ("gen_pass", "fast_pass", "plane") for t in ("double", "float")]
SOURCES += [(f"{s}.cu", f"{s}.o", ()) for s in ("engine_f32", "engine_f64", "noalloc", "capi", "probe")]
SOURCES += [("stage_radix.cu", f"stage_{t}_{p}.o", (f"-DLDDMM_STAGE_T={t}", f"-DLDDMM_STAGE_P={p}"))
            for t, ps in (("float", (6, 5, 4, 3)), ("double", (10, 9, 8, 6, 5, 4))) for p in ps]
SOURCES += [("stage_length.cu", f"stage_n{n}.o", (f"-DLDDMM_STAGE_N={n}",)) for n in stage_lengths()]
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
    objs = []
    cmds = []
    for src, name, defines in SOURCES:
        obj = os.path.join(BUILD_DIR, name)
        objs.append(obj)
        cmd = [nvcc, *_flags(extra_flags), *defines, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), flush=True)
        cmds.append(cmd)
    # one compiler per core at a time
    failed = []
    run = lambda cmd: subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    with ThreadPoolExecutor(os.cpu_count() or 1) as ex:
        for (src, name, _), p in zip(SOURCES, ex.map(run, cmds)):
            if p.returncode != 0 or verbose:
                sys.stderr.write(p.stdout.decode(errors="replace"))
            if p.returncode != 0:
                failed.append(name)
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
