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
import warnings
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
HEADER = os.path.join(os.path.dirname(HERE), "include", "mikv.h")
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
    files += [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    return files + [HEADER]


def pycall_path(debug: bool = False) -> str:
    """The extension module of this interpreter (its ABI is part of the name: another one builds its own)."""
    return os.path.join(OUT_DIR_DEBUG if debug else OUT_DIR, "mikv_pycall" + sysconfig.get_config_var("EXT_SUFFIX"))


def _pycall_tools():
    """(C compiler, folder of Python's headers), or None where one is missing."""
    include = sysconfig.get_paths()["include"]
    cc = shutil.which("gcc") or shutil.which("cc")
    return (cc, include) if cc and os.path.exists(os.path.join(include, "Python.h")) else None


def _build_pycall(debug: bool) -> None:
    """The optional extension module: without the tools, or if it does not compile, there is none (and no stale one), and
    the calls go through ctypes."""
    out, tools = pycall_path(debug), _pycall_tools()
    if tools:
        tmp = out + f".tmp{os.getpid()}"
        cmd = [tools[0], "-O2", "-std=c11", "-shared", "-fPIC", "-Wall", "-I", tools[1], os.path.join(CSRC, PYCALL), "-o", tmp]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode == 0:
            os.replace(tmp, out)
            return
        warnings.warn(f"{tools[0]} failed on {PYCALL}, the decode calls go through ctypes:\n{r.stdout}\n{r.stderr}")
    if os.path.exists(out):
        os.unlink(out)


def _current(target: str, inputs) -> bool:
    return os.path.exists(target) and all(os.path.getmtime(f) <= os.path.getmtime(target) for f in inputs)


def _lib_current(debug: bool) -> bool:
    return _current(LIB_DEBUG if debug else LIB, _inputs())


def _pycall_current(debug: bool) -> bool:
    return not _pycall_tools() or _current(pycall_path(debug), [os.path.join(CSRC, PYCALL), HEADER])


def up_to_date(debug: bool = False) -> bool:
    return _lib_current(debug) and _pycall_current(debug)


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    lib, out_dir = (LIB_DEBUG, OUT_DIR_DEBUG) if debug else (LIB, OUT_DIR)
    os.makedirs(out_dir, exist_ok=True)
    if force or not _pycall_current(debug):
        _build_pycall(debug)
    if not force and _lib_current(debug):
        return lib
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
