"""Builds the CUDA library paper_2010_14298_gb300/_lib/libfqt.so for sm_103a.

Each translation unit is compiled by nvcc in parallel, then linked into one
shared object with a plain C ABI (include/fqt.h).  The Python binding's native
marshalling (csrc/fqt_py.c) is a small extension module linked against it, named
for the interpreter it is built for; where it cannot be built (no C compiler, no
Python.h) the binding marshals through ctypes.  Run as a script or call
``build()``; what is up to date is not rebuilt.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys
import sysconfig
import warnings

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIBDIR = os.path.join(PKG, "_lib")
LIB = os.path.join(LIBDIR, "libfqt.so")
# another interpreter finds no extension module under its own name
PYEXT = os.path.join(LIBDIR, "_fqt_py" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
SOURCES = ["fqt_quant.cu", "fqt_codes.cu", "fqt_group.cu", "fqt_gemm.cu", "fqt_gemm_pair.cu", "fqt_conv.cu",
           "fqt_api.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC",
         "-Xcompiler", "-fvisibility=hidden", "--expt-relaxed-constexpr"]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _fresh(target, inputs) -> bool:
    if not os.path.exists(target):
        return False
    t = os.path.getmtime(target)
    inputs = [*inputs, os.path.join(INCLUDE, "fqt.h"), os.path.abspath(__file__)]
    return all(os.path.getmtime(f) <= t for f in inputs)


def library_up_to_date() -> bool:
    return _fresh(LIB, [os.path.join(CSRC, s) for s in SOURCES]
                  + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))])


def extension_up_to_date() -> bool:
    return _fresh(PYEXT, [os.path.join(CSRC, "fqt_py.c")])


def up_to_date() -> bool:
    return library_up_to_date() and extension_up_to_date()


def build_extension() -> bool:
    """Builds the extension module; a warning and False where it cannot be."""
    tmp = PYEXT + f".tmp{os.getpid()}"
    cmd = [shutil.which("gcc") or shutil.which("cc") or "gcc", "-O2", "-std=c11", "-shared",
           "-fPIC", "-I", sysconfig.get_paths()["include"], "-I", INCLUDE,
           os.path.join(CSRC, "fqt_py.c"), "-o", tmp, "-L", LIBDIR, "-l:libfqt.so",
           "-Wl,-rpath,$ORIGIN"]
    try:
        r = subprocess.run(cmd, capture_output=True, text=True)
        why = (r.stdout + r.stderr or f"exit status {r.returncode}") if r.returncode else ""
    except OSError as e:
        why = str(e)
    if why:
        if os.path.exists(PYEXT):  # of other sources: not to be loaded
            os.remove(PYEXT)
        warnings.warn("the Python extension module was not built, the binding marshals through "
                      f"ctypes:\n{why}", RuntimeWarning, stacklevel=2)
        return False
    os.replace(tmp, PYEXT)
    return True


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(LIBDIR, exist_ok=True)
    if force or not library_up_to_date():
        _build_library(verbose)
    if force or not extension_up_to_date():
        build_extension()
    return LIB


def _build_library(verbose: bool) -> None:
    nvcc = _nvcc()
    objs = []

    def compile_one(src):
        obj = os.path.join(LIBDIR, os.path.splitext(src)[0] + ".o")
        cmd = [nvcc, *ARCH, *FLAGS, "-I", INCLUDE, "-I", CSRC, "-c",
               os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), flush=True)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        return obj

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc, *ARCH, "-shared", "-o", tmp, *objs, "-lcudart",
           "-Xlinker", "-rpath", "-Xlinker", "/usr/local/cuda/lib64"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
