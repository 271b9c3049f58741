"""Compiles a CUDA source against the library's device headers into a shared object, so that
a test can run single operations of the kernels over many values."""
import ctypes
import os
import subprocess

from paper_2201_12404_gb300 import build


def load(directory, source):
    src, lib = os.path.join(directory, "ops.cu"), os.path.join(directory, "libops.so")
    with open(src, "w") as f:
        f.write(source)
    res = subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                          "-I", os.path.join(build.ROOT, "include"), "-o", lib, src],
                         capture_output=True, text=True, timeout=600)
    assert res.returncode == 0, res.stdout + res.stderr
    return ctypes.CDLL(lib)
