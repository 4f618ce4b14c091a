"""Builds a few lines of C++ that include the library's internal header, as a shared library for ctypes:
host-side tests of the rules the kernels and the host share."""
import ctypes
import os
import subprocess

from paper_1509_08267_gb300 import _build


def compile_shim(tmp_path, body: str) -> ctypes.CDLL:
    src, so = tmp_path / "shim.cpp", tmp_path / "shim.so"
    src.write_text('#include "gc_internal.h"\n' + body)
    cuda = os.path.dirname(os.path.dirname(_build.nvcc()))
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", _build.CSRC,
                    "-I", os.path.join(_build.ROOT, "include"), "-I", os.path.join(cuda, "include"),
                    str(src), "-o", str(so)], check=True, capture_output=True, text=True)
    return ctypes.CDLL(str(so))
