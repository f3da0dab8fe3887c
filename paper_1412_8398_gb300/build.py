"""Build the in-tree CUDA library ``_build/libfftls.so`` for sm_103a with nvcc.

The translation units are compiled in parallel and linked into a shared
library exporting the C ABI of ``include/fftls.h`` and ``include/fftls_nn.h``.  The build is skipped
when the library is newer than every source and header.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(BUILD, "libfftls.so")
SOURCES = ["fftls_kernels_x32.cu", "fftls_kernels_x64.cu", "fftls_kernels_y32.cu", "fftls_kernels_y64.cu",
           "fftls_kernels_z32.cu", "fftls_kernels_z64.cu", "fftls_kernels_x32g.cu", "fftls_kernels_x64g.cu",
           "fftls_kernels_y32g.cu", "fftls_kernels_y64g.cu", "fftls_kernels_z32g.cu", "fftls_kernels_z64g.cu",
           "fftls_kernels_t32.cu", "fftls_kernels_t64.cu", "fftls_kernels_yr32.cu", "fftls_kernels_zr32.cu",
           "fftls_solver.cu", "fftls_nn.cu", "fftls_nn_tc.cu",
           "fftls_nn_tc_conv1.cu", "fftls_nn_tc_conv3.cu", "fftls_nn_tc_conv3p.cu",
           "fftls_nn_tc_wgrad1.cu", "fftls_nn_tc_wgrad3.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc_path() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libfftls")


def _inputs():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files += [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    files.append(os.path.abspath(__file__))
    return files


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(f) <= t for f in _inputs())


def build(force: bool = False, verbose: bool = False, extra_flags=None) -> str:
    """Compile and link the library; returns its path."""
    if not force and up_to_date():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    nvcc = nvcc_path()
    flags = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-pthread", "-I", INCLUDE,
                    "-I", CSRC]
    if extra_flags:
        flags += list(extra_flags)

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.splitext(src)[0] + ".o")
        cmd = [nvcc, "-c", os.path.join(CSRC, src), "-o", obj] + flags
        p = subprocess.run(cmd, capture_output=True, text=True)
        if p.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{p.stdout}\n{p.stderr}")
        if verbose and (p.stdout or p.stderr):
            sys.stderr.write(p.stdout + p.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + ".tmp"
    cmd = [nvcc, "-shared", "-o", tmp] + objs + ARCH + ["--cudart", "static", "-lpthread"]
    p = subprocess.run(cmd, capture_output=True, text=True)
    if p.returncode != 0:
        raise RuntimeError(f"link failed:\n{p.stdout}\n{p.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
