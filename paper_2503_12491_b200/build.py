"""Builds libcake.so (sm_100a only, nvcc) and the binding's native half (_cake_py.*.so, g++) in-tree.

    python -m paper_2503_12491_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig
from typing import List

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB = os.path.join(PKG, "libcake.so")
PY_SOURCE = os.path.join(CSRC, "py_args.cpp")

SOURCES = ["cake_api.cu", "score_simt.cu", "score_tc.cu", "cascade.cu", "compact.cu",
           "decode.cu", "quant.cu", "select_static.cu"]


def binding_path() -> str:
    """The binding's native half for this interpreter and this torch: its file name has both, since it is
    built against either's ABI and another one's must not be loaded."""
    import torch
    return os.path.join(PKG, f"_cake_py.torch-{torch.__version__}.{sysconfig.get_config_var('SOABI')}.so")


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _inputs() -> List[str]:
    files = [os.path.join(CSRC, s) for s in SOURCES]
    files += [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    files += [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    return files


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(f) > t for f in _inputs())


def _run(cmd: List[str], what: str, verbose: bool) -> None:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError(f"compiler failed building {what}")


def build_binding(force: bool = False, verbose: bool = False) -> None:
    """Compiles the native half of binding.py against this interpreter and its torch."""
    deps, out = [PY_SOURCE, os.path.join(INCLUDE, "cake.h")], binding_path()
    if not force and os.path.exists(out) and all(os.path.getmtime(f) <= os.path.getmtime(out) for f in deps):
        return
    import torch
    home = os.path.dirname(torch.__file__)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_nvcc()))), "include")
    libs = os.path.join(home, "lib")
    _run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC",
          f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-I", INCLUDE,
          "-I", sysconfig.get_paths()["include"], "-isystem", os.path.join(home, "include"), "-isystem", cuda,
          PY_SOURCE, "-o", out, "-L", libs, f"-Wl,-rpath,{libs}", "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10",
          "-lc10_cuda", "-ldl"], os.path.basename(out), verbose)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles every CUDA source for sm_100a into one shared library, and the binding's native half."""
    build_binding(force, verbose)
    if not force and not is_stale():
        return LIB
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3",
           "-std=c++17", "--shared", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC,
           "--threads", "4"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", LIB]
    _run(cmd, "libcake.so", verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
