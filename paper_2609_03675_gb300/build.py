"""Builds libcofie_ngff.so (the CUDA kernels and the C ABI) in-tree.

nvcc compiles each translation unit for sm_103a only (no PTX for other
architectures), in parallel, then links a shared library next to this file.
Objects go to ``_build/`` (git-ignored). No CPU fallback is built.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
REPO = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(REPO, "include")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libcofie_ngff.so")
SOURCES = ["ngff_api.cu", "ngff_hist.cu", "ngff_features.cu", "ngff_select.cu", "ngff_chain.cu", "ngff_lazy.cu",
           "ngff_finalize.cu",
           "ngff_static.cu", "qer.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _flags(extra=()):
    return ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-O2", "-I", INCLUDE, "-I", CSRC,
                   *extra]


def _inputs():
    headers = ["ngff_common.cuh", "ngff_device.cuh"]
    files = ([os.path.join(CSRC, s) for s in SOURCES + headers]
             + [os.path.join(INCLUDE, "cofie_ngff.h"), __file__])
    return files


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(f) <= t for f in _inputs())


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False, defines=(), out: str | None = None,
          build_dir: str | None = None) -> str:
    """Compiles the library. ``defines`` (e.g. ["COFIE_K1_STAGES=6"]) and
    ``out``/``build_dir`` build a variant elsewhere without touching the default."""
    lib_path = out or LIB
    bdir = build_dir or BUILD
    if not force and not defines and out is None and up_to_date():
        return LIB
    os.makedirs(bdir, exist_ok=True)
    cc = nvcc()
    extra = (["-Xptxas", "-v"] if ptxas_info else []) + [f"-D{d}" for d in defines]

    def compile_one(src):
        obj = os.path.join(bdir, os.path.splitext(src)[0] + ".o")
        cmd = [cc, *_flags(extra), "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose or ptxas_info:
            sys.stderr.write(r.stdout + r.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = lib_path + f".tmp{os.getpid()}"
    cmd = [cc, *ARCH, "-shared", "-Xcompiler", "-fPIC", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, lib_path)
    return lib_path


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv))
