"""Compile the library's host-compilable headers (csrc/*.cuh whose functions are __host__ __device__) with g++ and load
the result, so that their arithmetic is tested without a GPU."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1311_4627_gb300", "csrc")


def cuda_home():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("the CUDA toolkit's headers are needed")
    return os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))


def compile_host(tmp, source):
    src, lib = os.path.join(tmp, "host.cpp"), os.path.join(tmp, "libhost.so")
    with open(src, "w") as f:
        f.write(source)
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC,
                    "-I", os.path.join(cuda_home(), "include"), src, "-o", lib], check=True)
    return ctypes.CDLL(lib)
