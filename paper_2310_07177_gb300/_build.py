"""Build libosd.so (the CUDA kernels behind include/osd.h) in-tree with nvcc,
and the binding, the Python calls in native code over it, with g++.

One translation unit per source file, compiled in parallel (the kernels for
sm_103a only), then linked into ``paper_2310_07177_gb300/libosd.so`` against the
shared CUDA runtime.  Rebuilds only when a source or header is newer than the
libraries.
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import shutil
import subprocess
import sysconfig

import torch

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD_DIR = os.path.join(PKG, "_build")
LIB_PATH = os.path.join(PKG, "libosd.so")
BINDING_SRC = os.path.join(CSRC, "osd_binding.cpp")
# compiled against torch's C++ and Python's C interface, of which its name says the versions:
# one of another torch or Python is neither taken for current nor loaded
BINDING_PATH = os.path.join(PKG, f"_binding-{torch.__version__}-{sysconfig.get_config_var('SOABI')}.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]


def nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: the CUDA 13 toolkit is required to build libosd.so")
    return exe


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _inputs():
    return _sources() + [BINDING_SRC] + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.hpp")) + \
        glob.glob(os.path.join(INCLUDE, "*.h"))


def up_to_date() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(BINDING_PATH):
        return False
    t = min(os.path.getmtime(LIB_PATH), os.path.getmtime(BINDING_PATH))
    return all(os.path.getmtime(f) <= t for f in _inputs())


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False) -> str:
    """Compile every .cu under csrc/ and the binding, link libosd.so and the binding;
    returns the path of the former."""
    if not force and up_to_date():
        return LIB_PATH
    os.makedirs(BUILD_DIR, exist_ok=True)
    exe = nvcc()
    extra = ["-Xptxas", "-v"] if ptxas_info else []

    def compile_one(src):
        obj = os.path.join(BUILD_DIR, os.path.basename(src) + ".o")
        cmd = [exe, *ARCH, *NVCC_FLAGS, *extra, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose or ptxas_info:
            print(r.stdout + r.stderr)
        return obj

    tdir = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(exe)))
    binding_obj = os.path.join(BUILD_DIR, "osd_binding.cpp.o")

    def compile_binding():
        cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-I", INCLUDE, "-I", sysconfig.get_paths()["include"],
               "-I", os.path.join(tdir, "include"), "-I", os.path.join(cuda, "include"), "-c", BINDING_SRC,
               "-o", binding_obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"g++ failed on {BINDING_SRC}:\n{r.stdout}\n{r.stderr}")

    with cf.ThreadPoolExecutor(max_workers=max(1, min(8, os.cpu_count() or 1))) as ex:
        binding = ex.submit(compile_binding)
        objs = list(ex.map(compile_one, _sources()))
        binding.result()
    tmp = LIB_PATH + f".tmp{os.getpid()}"
    cmd = [exe, *ARCH, "-shared", "-cudart", "shared", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link of libosd.so failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB_PATH)
    tmp = BINDING_PATH + f".tmp{os.getpid()}"
    cmd = ["g++", "-shared", "-o", tmp, binding_obj, "-L", PKG, "-l:" + os.path.basename(LIB_PATH), "-Wl,-rpath,$ORIGIN",
           "-L", os.path.join(tdir, "lib"),
           "-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10_cuda", "-lc10"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link of the binding failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, BINDING_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, ptxas_info=True))
