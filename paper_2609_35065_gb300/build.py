"""Build ``libkvs.so`` (the C-ABI library) in-tree with nvcc for sm_103a, and the Python
binding's marshalling extension beside it.

``python -m paper_2609_35065_gb300.build`` or ``build_library()``.  Both land in
``paper_2609_35065_gb300/_build/`` (git-ignored) and are rebuilt when a source or the
public header is newer.  The extension is optional: where it cannot be built or loaded (no
Python headers, no C compiler, a folder that cannot be written) the binding marshals with
numpy and ctypes, after a warning.
"""
from __future__ import annotations

import importlib.util
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
OUT_DIR = os.path.join(PKG, "_build")
LIB = os.path.join(OUT_DIR, "libkvs.so")
SOURCES = [os.path.join(CSRC, f) for f in ("kvs_kernels.cu", "kvs_api.cpp", "kvs_noalloc.cu", "kvs_fp8.cu",
                                           "kvs_tier.cpp")]
DEPS = SOURCES + [os.path.join(CSRC, "kvs_internal.h"), os.path.join(CSRC, "kvs_async.cuh"),
                  os.path.join(CSRC, "kvs_job.cuh"), os.path.join(INCLUDE, "kvs.h")]
ARCH = "-gencode=arch=compute_103a,code=sm_103a"


PYCALL_SOURCE = os.path.join(CSRC, "kvs_pycall.c")
PYCALL = os.path.join(OUT_DIR, "kvs_pycall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))


def _has_python_headers() -> bool:
    return os.path.exists(os.path.join(sysconfig.get_paths()["include"], "Python.h"))


def nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libkvs.so")


def command(out: str = LIB, extra: list[str] | None = None) -> list[str]:
    return [nvcc(), "-O3", "-lineinfo", "-std=c++17", ARCH, "-Xcompiler", "-fPIC,-O2,-Wall",
            "-shared", "--threads", "4", "-I", INCLUDE, *SOURCES, "-o", out, *(extra or [])]


def pycall_command(out: str = PYCALL) -> list[str]:
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        raise RuntimeError("a C compiler is required to build the binding's extension")
    return [cc, "-O2", "-Wall", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], "-I", INCLUDE,
            PYCALL_SOURCE, "-o", out]


def _older(out: str, deps) -> bool:
    if not os.path.exists(out):
        return True
    t = os.path.getmtime(out)
    return any(os.path.getmtime(d) > t for d in deps)


def stale(out: str = LIB) -> bool:
    return _older(out, DEPS)


def pycall_stale() -> bool:
    return _older(PYCALL, [PYCALL_SOURCE, os.path.join(INCLUDE, "kvs.h")])


def _usable_pycall(force: bool = False, verbose: bool = False) -> bool:
    """Whether an extension no older than its sources is there, built now if need be (or forced).
    One that is older and cannot be rebuilt is not usable: the structs it fills may have changed."""
    try:
        if force or pycall_stale():
            if not _has_python_headers():
                return False
            build_pycall(verbose)
        return True
    except (OSError, RuntimeError, subprocess.SubprocessError) as e:
        warnings.warn(f"the binding's extension cannot be built, arguments are marshalled with numpy: {e}",
                      RuntimeWarning, stacklevel=3)
        return False


def load_pycall():
    """The extension's ``call``, or None where it cannot be built or loaded."""
    if not _usable_pycall():
        return None
    try:
        spec = importlib.util.spec_from_file_location("kvs_pycall", PYCALL)
        mod = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(mod)
    except ImportError as e:
        warnings.warn(f"the binding's extension cannot be loaded, arguments are marshalled with numpy: {e}",
                      RuntimeWarning, stacklevel=2)
        return None
    return mod.call


def build_pycall(verbose: bool = False) -> None:
    os.makedirs(OUT_DIR, exist_ok=True)
    tmp = PYCALL + f".{os.getpid()}.tmp"
    cmd = pycall_command(tmp)
    if verbose:
        print(" ".join(cmd), file=sys.stderr)
    subprocess.run(cmd, check=True)
    os.replace(tmp, PYCALL)


def build_library(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OUT_DIR, exist_ok=True)
    _usable_pycall(force, verbose)
    if force or stale():
        tmp = LIB + f".{os.getpid()}.tmp"
        cmd = command(tmp)
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        subprocess.run(cmd, check=True)
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose=True))
