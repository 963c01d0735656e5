"""Build the CUDA library libpuro_fp8.so in-tree with nvcc for sm_103a.

Five translation units are compiled in parallel and linked into one shared
object with the CUDA runtime linked statically, so the library loads on a
machine without a GPU driver (only the first CUDA call needs one).  Beside it
the Python binding's native marshalling module _native.so is compiled and
linked against the installed torch (the library's entry points are handed to it).
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libpuro_fp8.so")
NATIVE = os.path.join(PKG, "_native.so")
BINDING = os.path.join(CSRC, "binding.cpp")
NATIVE_FOR = os.path.join(BUILD, "native_for.txt")  # what _native.so was compiled for
SOURCES = ["api.cu", "quantize.cu", "gemm.cu", "noalloc.cu", "muonh.cu"]
HEADERS = ["ptx.cuh", "internal.h", "quant_math.cuh"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
              "-Xcompiler", "-Wall", "--expt-relaxed-constexpr", "-I", INCLUDE, "-I", CSRC]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libpuro_fp8.so")


def native_for() -> str:
    """The torch and the interpreter that _native.so has to be compiled for: neither keeps
    its binary interface from one version to the next."""
    import torch

    return f"torch {torch.__version__}, {sys.implementation.cache_tag}"


def _stale() -> bool:
    if not all(os.path.exists(f) for f in (LIB, NATIVE, NATIVE_FOR)):
        return True
    with open(NATIVE_FOR) as f:
        if f.read() != native_for():
            return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(NATIVE))
    deps = [BINDING] + [os.path.join(CSRC, f) for f in SOURCES + HEADERS] + [os.path.join(INCLUDE, "puro_fp8.h"),
                                                                  os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile (if stale) and return the path of libpuro_fp8.so."""
    if not force and not _stale():
        return LIB
    nvcc = _nvcc()
    os.makedirs(BUILD, exist_ok=True)

    def compile_one(src: str) -> str:
        obj = os.path.join(BUILD, os.path.splitext(src)[0] + ".o")
        cmd = [nvcc, *ARCH, *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), flush=True)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose and (r.stdout or r.stderr):
            print(r.stdout, r.stderr, flush=True)
        return obj

    def compile_binding() -> str:
        import torch  # headers only: the module is compiled for the torch it is imported beside

        inc = os.path.join(os.path.dirname(torch.__file__), "include")
        obj = os.path.join(BUILD, "binding.o")
        cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden", "-Wall",
               f'-DPURO_NATIVE_FOR="{native_for()}"', "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI, "-isystem", inc, "-isystem",
               os.path.join(inc, "torch", "csrc", "api", "include"), "-isystem", sysconfig.get_paths()["include"],
               "-isystem", os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include"),
               "-I", INCLUDE, "-c", BINDING, "-o", obj]
        if verbose:
            print(" ".join(cmd), flush=True)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"g++ failed on binding.cpp:\n{r.stdout}\n{r.stderr}")
        return obj

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES) + 1) as ex:
        binding = ex.submit(compile_binding)
        objs = list(ex.map(compile_one, SOURCES))
        binding_obj = binding.result()
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc, *ARCH, "-shared", "-cudart", "static", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)

    import torch

    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = NATIVE + ".tmp.%d" % os.getpid()
    cmd = ["g++", "-shared", "-o", tmp, binding_obj, "-L", libs, "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link of the binding failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, NATIVE)
    with open(NATIVE_FOR, "w") as f:
        f.write(native_for())
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
