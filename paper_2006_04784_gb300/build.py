"""Build libfch.so (the CUDA path) in-tree for sm_103a.

Compiles each translation unit of csrc/ with nvcc in parallel and links them
into paper_2006_04784_gb300/_build/libfch.so. Only rebuilds what changed.
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_build")
LIB = os.path.join(OUT, "libfch.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
              "--expt-relaxed-constexpr"]


def nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libfch")


def _deps():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + [
        os.path.join(HERE, "..", "include", "fch.h")]


# fch_reg.cu holds the passes built for one (precision, grid size): one object each
REG_SRC = os.path.join(CSRC, "fch_reg.cu")
REG_TYPES = (("fch::df", "dfl"), ("double", "f64"), ("float", "f32"))
REG_LOGN = range(6, 12)


def _units():
    """(source, object name, extra flags) of every compilation, the longest first"""
    reg = [(REG_SRC, f"fch_reg_{sfx}_{l}.o", [f"-DFCH_T={t}", f"-DFCH_SUFFIX={sfx}", f"-DFCH_LOGN={l}"])
           for t, sfx in REG_TYPES for l in reversed(REG_LOGN)]
    rest = [(s, os.path.basename(s) + ".o", []) for s in sorted(glob.glob(os.path.join(CSRC, "*.cu"))) if s != REG_SRC]
    return rest + reg


def _compile(src: str, name: str, extra) -> str:
    obj = os.path.join(OUT, name)
    newest = max(os.path.getmtime(p) for p in _deps() + [src, __file__])
    if os.path.exists(obj) and os.path.getmtime(obj) >= newest:
        return obj
    tmp = obj + f".{os.getpid()}.tmp"
    cmd = [nvcc(), *ARCH, *NVCC_FLAGS, *extra, "-c", src, "-o", tmp]
    subprocess.check_call(cmd)
    os.replace(tmp, obj)
    return obj


def build(verbose: bool = False, extra=()) -> str:
    """Compile every CUDA source of the package; returns the library path."""
    os.makedirs(OUT, exist_ok=True)
    units = _units()
    extra = list(extra) + (["-Xptxas", "-v"] if verbose else [])
    with cf.ThreadPoolExecutor(max_workers=os.cpu_count() or 8) as ex:
        objs = list(ex.map(lambda u: _compile(u[0], u[1], u[2] + extra), units))
    newest = max(os.path.getmtime(o) for o in objs)
    if not os.path.exists(LIB) or os.path.getmtime(LIB) < newest:
        tmp = LIB + f".{os.getpid()}.tmp"
        subprocess.check_call([nvcc(), *ARCH, "-shared", "-o", tmp, *objs])
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(verbose="-v" in sys.argv))
