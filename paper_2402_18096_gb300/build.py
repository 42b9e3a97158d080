"""Build libmikv.so (the CUDA kernels + C ABI) for sm_103a, in-tree under ``_build/``.

Each translation unit compiles in parallel with nvcc; the objects are linked into one shared library.
``build(debug=True)`` builds the checked variant (-DMIKV_DEBUG: kernels record out-of-range indices in a status
word, see include/mikv.h) as ``_build_debug/libmikv_debug.so``.
Usage: ``python -m paper_2402_18096_gb300.build [--debug]`` or ``build()`` from Python.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(OUT_DIR, "libmikv.so")
OUT_DIR_DEBUG = os.path.join(HERE, "_build_debug")
LIB_DEBUG = os.path.join(OUT_DIR_DEBUG, "libmikv_debug.so")
SOURCES = ["mikv_attn_h16.cu", "mikv_attn_h8.cu", "mikv_attn_h4.cu", "mikv_attn_h2.cu", "mikv_attn_kch.cu",
           "mikv_attention.cu",
           "mikv_quant.cu", "mikv_policy.cu", "mikv_step.cu", "mikv_prefill.cu", "mikv_abi.cu"]
PYCALL = "mikv_pycall.c"  # the binding's decode-path calls as an extension module (where Python's headers are installed)
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]
# a register spilled in the kernels that load from tensor memory is an error (see tmem_ld32)
SOURCE_FLAGS = {"mikv_prefill.cu": ["-Xptxas", "-warn-spills,-Werror"]}


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libmikv")


def source_flags(src: str, debug: bool = False) -> list:
    return NVCC_FLAGS + SOURCE_FLAGS.get(src, []) + (["-DMIKV_DEBUG"] if debug else [])


def _inputs():
    files = [os.path.join(CSRC, s) for s in SOURCES]
    files += [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h", ".c"))]
    files.append(os.path.join(os.path.dirname(HERE), "include", "mikv.h"))
    return files


def pycall_path(debug: bool = False) -> str:
    return os.path.join(OUT_DIR_DEBUG if debug else OUT_DIR, "mikv_pycall.so")


def _build_pycall(debug: bool) -> None:
    """The extension module, or none (and no stale one) without Python's headers or a C compiler."""
    out = pycall_path(debug)
    include = sysconfig.get_paths()["include"]
    gcc = shutil.which("gcc") or shutil.which("cc")
    if not gcc or not os.path.exists(os.path.join(include, "Python.h")):
        if os.path.exists(out):
            os.unlink(out)
        return
    tmp = out + f".tmp{os.getpid()}"
    cmd = [gcc, "-O2", "-std=c11", "-shared", "-fPIC", "-Wall", "-I", include, os.path.join(CSRC, PYCALL), "-o", tmp]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"{gcc} failed on {PYCALL}:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, out)


def up_to_date(debug: bool = False) -> bool:
    lib = LIB_DEBUG if debug else LIB
    if not os.path.exists(lib):
        return False
    t = os.path.getmtime(lib)
    return all(os.path.getmtime(f) <= t for f in _inputs())


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    lib, out_dir = (LIB_DEBUG, OUT_DIR_DEBUG) if debug else (LIB, OUT_DIR)
    if not force and up_to_date(debug):
        return lib
    os.makedirs(out_dir, exist_ok=True)
    nvcc = _nvcc()

    def compile_one(src):
        obj = os.path.join(out_dir, os.path.splitext(src)[0] + ".o")
        cmd = [nvcc, *ARCH, *source_flags(src, debug), "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose and (r.stdout or r.stderr):
            print(r.stdout, r.stderr, file=sys.stderr)
        return obj

    _build_pycall(debug)
    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = lib + f".tmp{os.getpid()}"
    cmd = [nvcc, *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, debug="--debug" in sys.argv))
