"""Builds the C-ABI shared library (libprepack_b200.so) in-tree with nvcc for sm_100a, and the Python
module over it (_native)."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libprepack_b200.so")
MODULE_PATH = os.path.join(PKG_DIR, "_native" + sysconfig.get_config_var("EXT_SUFFIX"))
SOURCES = ["pp_host.cpp", "pp_api.cu", "pp_rope.cu", "pp_attention.cu", "pp_unpack.cu", "pp_unpack_static.cu",
           "pp_tensorize.cu", "pp_decode.cu"]
MODULE_SOURCE = "pp_python.cpp"
HEADERS = ["pp_internal.h", "pp_device_once.h", os.path.join("..", "..", "include", "pp.h")]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; the prepack-b200 library needs the CUDA toolkit to build")


def is_stale() -> bool:
    for path, sources in ((LIB_PATH, SOURCES), (MODULE_PATH, [MODULE_SOURCE])):
        if not os.path.exists(path):
            return True
        t = os.path.getmtime(path)
        if any(os.path.getmtime(os.path.join(CSRC, s)) > t for s in sources + HEADERS):
            return True
    return False


def _run(cmd: list, verbose: bool) -> None:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    if verbose:
        sys.stderr.write(res.stderr)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source for sm_100a into one shared library; returns its path."""
    if not force and not is_stale():
        return LIB_PATH
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-Xcompiler", "-fPIC", "-shared", "-x", "cu"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES]
    cmd += ["-o", LIB_PATH]
    _run(cmd, verbose)
    import numpy
    _run([_nvcc(), "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", sysconfig.get_paths()["include"],
          "-I", numpy.get_include(), os.path.join(CSRC, MODULE_SOURCE), "-o", MODULE_PATH, "-L", PKG_DIR,
          "-l:" + os.path.basename(LIB_PATH), "-Xlinker", "-rpath=$ORIGIN"], verbose)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
