"""In-tree build of libkeyless.so for sm_103a (GB300) with nvcc.

Each translation unit under ``csrc/`` is compiled in parallel to an object file, then the
objects are linked into ``_build/libkeyless.so`` with the CUDA runtime linked statically, so
the library has no dependency beyond the driver; the binding's C module
(``csrc/kl_python.c``) is compiled next to it, for the interpreter that builds it. Each of the
two is rebuilt only when one of its own sources is newer. Without Python's C headers the module is
left out (and the binding goes through ctypes).
"""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "libkeyless.so")
PYSRC = os.path.join(CSRC, "kl_python.c")
# named for the interpreter, as extension modules are: another Python builds its own beside it
PYMOD = os.path.join(BUILD, "_keyless" + sysconfig.get_config_var("EXT_SUFFIX"))

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
              "-I", INCLUDE, "-I", CSRC]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def python_headers() -> str | None:
    """The folder of Python.h, or None where Python's C headers are not installed."""
    paths = sysconfig.get_paths()
    for d in (paths["include"], paths["platinclude"]):
        if os.path.exists(os.path.join(d, "Python.h")):
            return d
    return None


def _stale(target: str, deps: list[str]) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(p) > os.path.getmtime(target) for p in deps)


def build(force: bool = False, verbose: bool = False, extra_flags: list[str] | None = None) -> str:
    """Build what is out of date: libkeyless.so for sm_103a (its path is returned) and the Python module."""
    headers = glob.glob(os.path.join(INCLUDE, "*.h"))
    if force or _stale(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + headers):
        _build_library(verbose, extra_flags)
    include = python_headers()
    if include and (force or _stale(PYMOD, [PYSRC] + headers)):
        _build_module(include)
    return LIB


def _build_library(verbose: bool, extra_flags: list[str] | None) -> None:
    """Compile every CUDA source for sm_103a and link libkeyless.so."""
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()
    flags = NVCC_FLAGS + (extra_flags or [])

    def compile_one(src: str) -> str:
        obj = os.path.join(BUILD, os.path.basename(src).replace(".cu", ".o"))
        cmd = [cc, *ARCH, *flags, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {os.path.basename(src)}:\n{r.stdout}\n{r.stderr}")
        if verbose and (r.stdout or r.stderr):
            print(r.stdout + r.stderr)
        return obj

    with ThreadPoolExecutor(max(1, min(len(sources()), os.cpu_count() or 1))) as ex:
        objs = list(ex.map(compile_one, sources()))
    tmp = LIB + ".tmp"
    cmd = [cc, *ARCH, "-shared", "-cudart", "static", *objs, "-o", tmp]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)


def _build_module(include: str) -> None:
    """The binding's Python module (host C; bound to the library at run time)."""
    os.makedirs(BUILD, exist_ok=True)
    tmp = PYMOD + ".tmp"
    cmd = [os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I", INCLUDE,
           "-I", include, PYSRC, "-o", tmp]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"building the Python module failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, PYMOD)


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose=True))
