"""Compiles a test's own CUDA source against the library's device headers."""
import ctypes
import os
import subprocess

from paper_2103_07210_gb300 import ftgcr

CSRC = os.path.join(os.path.dirname(os.path.abspath(ftgcr.__file__)), "csrc")


def compile_cuda(source: str, directory) -> ctypes.CDLL:
    """A shared library of `source`, compiled with the library's own flags."""
    src, out = os.path.join(str(directory), "unit.cu"), os.path.join(str(directory), "unit.so")
    with open(src, "w") as f:
        f.write(source)
    subprocess.check_call(["nvcc"] + ftgcr.NVCC_FLAGS + ["-shared", "-I", CSRC, "-o", out, src])
    return ctypes.CDLL(out)
