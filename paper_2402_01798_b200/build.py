"""Build libtq.so (the CUDA kernels + C ABI, nvcc for sm_100a) and the Python marshalling module, in-tree."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libtq.so")
NATIVE = os.path.join(PKG, "_tq_python" + sysconfig.get_config_var("EXT_SUFFIX"))
NATIVE_SOURCE = os.path.join(CSRC, "tq_python.cpp")
NATIVE_TORCH = os.path.join(PKG, "_tq_python.torch")       # the torch version that the module was built against: its C++ interface changes
SOURCES = ["tq_api.cu", "tq_stats.cu", "tq_compress.cu", "tq_compress_lut.cu", "tq_decompress.cu", "tq_params.cu"]
HEADERS = ["tq_aggregation_plan.h", "tq_device.cuh", "tq_launch.h", "tq_lut.cuh"]

NVCC_FLAGS = [
    "-std=c++17", "-O3", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
    "-fmad=false",                      # no implicit fused multiply-add: code decisions are one rounding per op
    "-Xcompiler", "-fPIC,-ffp-contract=off",
    "-cudart", "static",
]


def _stale(target: str, sources) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in [*sources, os.path.join(ROOT, "include", "tq.h"), __file__])


def _run(cmd, verbose: bool, what: str) -> None:
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError(f"building {what} failed")


def native_torch():
    """The torch version that the marshalling module was built against, None if that was not written down."""
    if not os.path.exists(NATIVE_TORCH):
        return None
    with open(NATIVE_TORCH) as f:
        return f.read().strip()


def build_native(force: bool = False, verbose: bool = False) -> str:
    """The marshalling module: C++ against torch's and Python's headers."""
    import torch
    if not force and native_torch() == torch.__version__ and not _stale(NATIVE, [NATIVE_SOURCE]):
        return NATIVE
    base = os.path.dirname(torch.__file__)
    inc = [os.path.join(base, "include"), os.path.join(base, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"), os.path.join(ROOT, "include")]
    tmp = NATIVE + f".tmp{os.getpid()}"
    libs = os.path.join(base, "lib")
    _run([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
          *[f"-I{p}" for p in inc], NATIVE_SOURCE, "-o", tmp, f"-L{libs}", f"-Wl,-rpath,{libs}", "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"],
         verbose, os.path.basename(NATIVE))
    os.replace(tmp, NATIVE)
    with open(NATIVE_TORCH, "w") as f:
        f.write(torch.__version__)
    return NATIVE


def build(force: bool = False, verbose: bool = False) -> str:
    build_native(force, verbose)
    if not force and not _stale(LIB, [os.path.join(CSRC, f) for f in SOURCES + HEADERS]):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + f".tmp{os.getpid()}"
    extra = os.environ.get("TQ_NVCC_EXTRA", "").split()
    cmd = [nvcc] + NVCC_FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) + [
        "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-shared", "-o", tmp,
    ] + [os.path.join(CSRC, f) for f in SOURCES]
    _run(cmd, verbose, "libtq.so")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
