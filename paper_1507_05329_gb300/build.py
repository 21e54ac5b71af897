"""Build the COLA CUDA library (libcola.so) in-tree for sm_103a with nvcc.

Each translation unit is compiled in parallel; the shared library links the CUDA runtime
statically so it does not depend on which libcudart the Python process already loaded.
"""

from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD_DIR = os.path.join(HERE, "_build")
LIB_PATH = os.path.join(HERE, "libcola.so")
CT_PARTS = 16   # parts of the per-length FFT kernels (fft_ct.cu), compiled in parallel
SOURCES = ["fft.cu", "fft_generic.cu", "particles.cu", "binning.cu", "adjoint.cu", "fof.cu", "cola_batch.cu",
           "cola_abi.cu", "cola_static.cu", "rng.cu", "host_cosmo.cpp"]
HEADERS = [os.path.join(CSRC, h) for h in ("cola_internal.h", "fft_core.cuh", "fft_ct.cuh", "fft_ops.h", "fft_plan.h")] + [
    os.path.join(ROOT, "include", "cola.h")]
# (source, object, extra flags) of every compilation
UNITS = [(s, s + ".o", []) for s in SOURCES] + [
    ("fft_ct.cu", f"fft_ct_{k}.o", [f"-DCOLA_CT_PART={k}"]) for k in range(CT_PARTS)]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I" + os.path.join(ROOT, "include"),
         f"-DCOLA_CT_PARTS={CT_PARTS}"]


def _nvcc() -> str:
    path = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(path):
        raise RuntimeError("nvcc not found: the COLA library needs the CUDA toolkit to build")
    return path


def _stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    deps = [os.path.join(CSRC, u[0]) for u in UNITS] + HEADERS + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every translation unit and link libcola.so; returns the library path."""
    if not force and not _stale():
        return LIB_PATH
    nvcc = _nvcc()
    os.makedirs(BUILD_DIR, exist_ok=True)

    def compile_one(unit) -> str:
        src, name, extra = unit
        obj = os.path.join(BUILD_DIR, name)
        cmd = [nvcc, *ARCH, *FLAGS, *extra, "-c", os.path.join(CSRC, src), "-o", obj]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{res.stdout}\n{res.stderr}")
        if verbose and (res.stdout or res.stderr):
            print(res.stdout + res.stderr)
        return obj

    with cf.ThreadPoolExecutor(max_workers=os.cpu_count() or 8) as ex:
        objs = list(ex.map(compile_one, UNITS))
    tmp = LIB_PATH + ".tmp"
    cmd = [nvcc, *ARCH, "-shared", "-cudart", "static", "-o", tmp, *objs]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link failed:\n{res.stdout}\n{res.stderr}")
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
