"""Builds libqvggt.so (CUDA kernels + C ABI, nvcc, sm_100a) and the Python call path in front of it (g++) in-tree."""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libqvggt.so")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")


def fastcall_path(torch_version: str = torch.__version__) -> str:
    """The extension module is bound to one Python and one torch: both are in its name, so that another one builds its own."""
    return os.path.join(_HERE, f"_qvggt_fastcall.{sysconfig.get_config_var('SOABI')}.torch-{torch_version}.so")


FASTCALL = fastcall_path()

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-fmad=false",            # bit-exact contract: no FMA contraction anywhere (FMAs are written explicitly)
    "-Xcompiler", "-fPIC", "-shared",
]


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target: str, deps: list[str]) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(f) > t for f in deps)


def _headers() -> list[str]:
    return glob.glob(os.path.join(INCLUDE, "*.h"))


def is_stale() -> bool:
    return (_stale(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + _headers())
            or _stale(FASTCALL, [os.path.join(CSRC, "fastcall.cpp")] + _headers()))


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + _headers()):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [nvcc, *NVCC_FLAGS, "-I", INCLUDE, "-o", tmp, *sources()]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    src = os.path.join(CSRC, "fastcall.cpp")
    if force or _stale(FASTCALL, [src] + _headers()):
        root = os.path.dirname(torch.__file__)
        tmp = FASTCALL + f".tmp{os.getpid()}"
        subprocess.check_call(
            [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
             "-I", INCLUDE, "-I", os.path.join(root, "include"), "-I", os.path.join(root, "include", "torch", "csrc", "api", "include"),
             "-I", "/usr/local/cuda/include", "-I", sysconfig.get_paths()["include"], "-o", tmp, src,
             "-L", _HERE, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN", "-L", os.path.join(root, "lib"),
             "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"])
        os.replace(tmp, FASTCALL)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
