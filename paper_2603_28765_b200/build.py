"""Builds the CUDA library in-tree with nvcc for sm_100a, and the host module that calls it with torch tensors."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB_PATH = os.path.join(_HERE, "libabs_b200.so")
SOURCES = [os.path.join(CSRC, "abs_b200.cu"), os.path.join(CSRC, "abs_gemm.cu")]
HEADERS = [os.path.join(CSRC, "abs_device.cuh"), os.path.join(CSRC, "abs_fast4.cuh"), os.path.join(CSRC, "abs_opt4.cuh"), os.path.join(CSRC, "abs_fastx.cuh"), os.path.join(CSRC, "abs_trans4.cuh"), os.path.join(CSRC, "abs_generic.cuh"), os.path.join(CSRC, "abs_rows.cuh"), os.path.join(CSRC, "abs_skinny.cuh"), os.path.join(CSRC, "abs_tc.cuh"), os.path.join(CSRC, "abs_pair.cuh"), os.path.join(CSRC, "abs_launch.h"), os.path.join(os.path.dirname(_HERE), "include", "abs_b200.h")]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-lineinfo", "-std=c++17",
    # bit-exactness: no implicit multiply-add contraction, IEEE division / sqrt, subnormals kept
    "-fmad=false", "-prec-div=true", "-prec-sqrt=true", "-ftz=false",
    "--shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
    "-cudart", "static", "-Xlinker", "-Bsymbolic",
]


CALL_SOURCES = [os.path.join(CSRC, "abs_call.cpp"), os.path.join(os.path.dirname(_HERE), "include", "abs_b200.h")]


def _older(target: str, sources) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in sources)


def needs_build() -> bool:
    return _older(LIB_PATH, SOURCES + HEADERS)


def call_path() -> str:
    """The host module of this interpreter and this torch: it is bound to the binary interface of both, so both are in its name."""
    import torch
    return os.path.join(_HERE, f"_abs_call-torch{torch.__version__}" + sysconfig.get_config_var("EXT_SUFFIX"))


def build_call(force: bool = False) -> str:
    """Compile the host module ``_abs_call`` (torch's C++ interface, no kernels) if it is missing or older than its sources."""
    path = call_path()
    if not force and not _older(path, CALL_SOURCES):
        return path
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    tmp = path + f".tmp{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    cmd += [x for p in inc for x in ("-isystem", p)] + ["-o", tmp, CALL_SOURCES[0], "-L" + os.path.join(root, "lib")]
    cmd += ["-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10", "-Wl,-rpath," + os.path.join(root, "lib")]
    subprocess.run(cmd, check=True)
    os.replace(tmp, path)
    return path


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile libabs_b200.so if it is missing or older than its sources (nvcc only: no torch needed). Returns its path."""
    if not force and not needs_build():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB_PATH + f".tmp{os.getpid()}"
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", tmp] + SOURCES
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
    print(build_call(force="--force" in sys.argv))
