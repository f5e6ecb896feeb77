"""In-tree build: nvcc -> paper_2505_18610_b200/libpmkvq.so (the CUDA library, sm_100a only) and the host compiler ->
paper_2505_18610_b200/_host_calls.so (the Python extension for the calls of the token loop, linked to the former)."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig

import torch

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "csrc", "pmkvq_api.cu")
LIB = os.path.join(HERE, "libpmkvq.so")
HOST_SRC = os.path.join(HERE, "csrc", "host_calls.cpp")
HOST_LIB = os.path.join(HERE, "_host_calls.so")
DEPS = [os.path.join(HERE, "csrc", f) for f in os.listdir(os.path.join(HERE, "csrc"))] + [
    os.path.join(os.path.dirname(HERE), "include", "pmkvq.h")]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
    "--fmad=true",        # contraction is allowed in the attention math; the quantizer uses *_rn intrinsics
    "-Xcompiler", "-fPIC", "-shared", "-Xptxas", "-v",
]


# The extension uses torch's C++ classes and CPython's structures, so it belongs to one torch and one Python; it carries this text.
HOST_FOR = f"built for torch {torch.__version__}, {sysconfig.get_config_var('SOABI')}"


def _stale(lib: str) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    return any(os.path.getmtime(d) > t for d in DEPS)


def _host_stale() -> bool:
    if _stale(HOST_LIB):
        return True
    with open(HOST_LIB, "rb") as f:
        return HOST_FOR.encode() not in f.read()


def needs_build() -> bool:
    return _stale(LIB) or _host_stale()


def _nvcc() -> str:
    return os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")   # a path, or a name to be found on PATH


def _cuda_home() -> str:
    return os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(_nvcc()) or _nvcc())))


def _build_host_calls() -> None:
    at = os.path.dirname(torch.__file__)
    include = [os.path.join(at, "include"), sysconfig.get_paths()["include"], os.path.join(_cuda_home(), "include")]
    cmd = ([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}", f'-DHOST_FOR="{HOST_FOR}"'] + ["-I" + i for i in include]
           + ["-o", HOST_LIB, HOST_SRC, "-L" + HERE, "-l:libpmkvq.so", "-Wl,-rpath,$ORIGIN", "-L" + os.path.join(at, "lib"),
              "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"])
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("the host compiler failed building _host_calls.so")


def _build_library(verbose: bool) -> None:
    cmd = [_nvcc()] + NVCC_FLAGS + ["-o", LIB, SRC]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("nvcc failed building libpmkvq.so")
    if verbose:
        sys.stderr.write(res.stderr)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale(LIB):
        _build_library(verbose)
    if force or _host_stale():
        _build_host_calls()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
