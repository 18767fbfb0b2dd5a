"""Builds the C-ABI shared library (libsegquant.so) from csrc/ with nvcc for sm_100a, in-tree."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
LIB_PATH = os.path.join(_HERE, "libsegquant.so")
OBJ_DIR = os.path.join(_HERE, "_build")
# (source, object, defines): the GEMM's kernel instantiations are spread over four units that compile side by side
UNITS = [(f, f.replace(".cu", ".o"), []) for f in ("api.cu", "calib.cu", "quantize.cu", "zero_point.cu", "gemm_tcgen05.cu")]
UNITS += [("gemm_tcgen05.cu", f"gemm_kind{k}_npol{n}.o", [f"-DSQ_GEMM_KIND={k}", f"-DSQ_GEMM_NPOL={n}"])
          for k in (0, 1) for n in (1, 2)]
CALLS_PATH = os.path.join(_HERE, "_calls.so")          # native module over the library, for torch tensors
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC"]


def _stale() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(CALLS_PATH):
        return True
    t = min(os.path.getmtime(LIB_PATH), os.path.getmtime(CALLS_PATH))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, "segquant.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles every translation unit (side by side) and links the shared library."""
    if not force and not _stale():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "nvcc")
    os.makedirs(OBJ_DIR, exist_ok=True)
    extra = ["-Xptxas", "-v"] if verbose else []

    def compile_one(unit):
        src, obj, defines = unit[0], os.path.join(OBJ_DIR, unit[1]), unit[2]
        subprocess.check_call([nvcc, *NVCC_FLAGS, *extra, *defines, "-I", INCLUDE, "-I", CSRC, "-c", os.path.join(CSRC, src), "-o", obj])
        return obj

    with ThreadPoolExecutor(max_workers=len(UNITS)) as pool:
        objs = list(pool.map(compile_one, UNITS))
    subprocess.check_call([nvcc, "-shared", "-cudart", "static", "-gencode", "arch=compute_100a,code=sm_100a",
                           "-o", LIB_PATH, *objs])
    build_calls(nvcc)
    return LIB_PATH


def build_calls(nvcc: str) -> None:
    """Compiles csrc/torch_calls.cpp against torch's headers and links it to the library beside it."""
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(nvcc) or "/usr/local/cuda/bin/nvcc"))), "include")
    include = [*cpp_extension.include_paths(), sysconfig.get_paths()["include"], cuda]
    subprocess.check_call([
        os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
        f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *[f for d in include for f in ("-isystem", d)],
        "-I", INCLUDE, os.path.join(CSRC, "torch_calls.cpp"), "-o", CALLS_PATH, "-L", _HERE, "-l:libsegquant.so",
        *[f for d in cpp_extension.library_paths() for f in ("-L", d)], "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda",
        "-Wl,-rpath,$ORIGIN"])


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
