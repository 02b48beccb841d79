"""Build libpic.so (the CUDA kernels and the C ABI) and _pic_native.so (the
Python binding's native part) in-tree for sm_103a.

Every translation unit under csrc/ is compiled in parallel, the .cu files with
nvcc, binding.cpp with the host compiler against the installed PyTorch's
headers; libpic.so is linked against the shared CUDA runtime (the copy PyTorch
has already loaded is reused), _pic_native.so against libpic.so and PyTorch.
No CMake, no torch extension machinery: a few seconds per file.
"""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
OUT_DIR = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libpic.so")
NATIVE = os.path.join(PKG, "_pic_native.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-cudart", "shared",
         "--expt-relaxed-constexpr", "-Xptxas", "-v"]


def _nvcc() -> str:
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libpic")
    return cand


def _compile(src: str) -> tuple[str, str]:
    obj = os.path.join(OUT_DIR, os.path.basename(src) + ".o")
    cmd = [_nvcc(), *ARCH, *FLAGS, "-c", src, "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
    return obj, r.stderr


def _cuda_lib() -> str:
    root = os.path.dirname(os.path.dirname(_nvcc()))
    return next((d for d in (os.path.join(root, "lib64"), os.path.join(root, "lib"))
                 if os.path.isdir(d)), os.path.join(root, "lib64"))


def _compile_binding() -> str:
    import torch
    troot = os.path.dirname(torch.__file__)
    inc = [os.path.join(troot, "include"), os.path.join(troot, "include/torch/csrc/api/include"),
           os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include"),
           sysconfig.get_paths()["include"]]
    obj = os.path.join(OUT_DIR, "binding.o")
    cmd = ["g++", "-O2", "-std=c++20", "-fPIC", "-fvisibility=hidden", *[f"-I{i}" for i in inc],
           "-c", os.path.join(CSRC, "binding.cpp"), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed on binding.cpp:\n{r.stdout}\n{r.stderr}")
    return obj


def _link_binding(obj: str) -> None:
    import torch
    tlib = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = NATIVE + ".tmp"
    cmd = ["g++", "-shared", "-o", tmp, obj, LIB, f"-L{tlib}", "-ltorch_python", "-ltorch_cpu",
           "-lc10", "-lc10_cuda", f"-L{_cuda_lib()}", "-lcudart", "-Wl,-rpath,$ORIGIN"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link of the binding failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, NATIVE)


def build(verbose: bool = False) -> str:
    """Compile and link; returns the library path.  Always rebuilds."""
    os.makedirs(OUT_DIR, exist_ok=True)
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    with ThreadPoolExecutor(max_workers=min(len(srcs) + 1, os.cpu_count() or 4)) as ex:
        binding = ex.submit(_compile_binding)
        results = list(ex.map(_compile, srcs))
    with open(os.path.join(OUT_DIR, "ptxas.log"), "w") as f:
        for (obj, log) in results:
            f.write(f"== {os.path.basename(obj)}\n{log}\n")
    tmp = LIB + ".tmp"
    cmd = [_nvcc(), *ARCH, "-shared", "-cudart", "shared", "-Xlinker", "-soname=libpic.so", "-o", tmp, *[o for o, _ in results]]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    _link_binding(binding.result())
    if verbose:
        print(f"built {LIB}", file=sys.stderr)
    return LIB


if __name__ == "__main__":
    build(verbose=True)
