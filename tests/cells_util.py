"""Builds tests/cells_protocol.cu, host code over the library's internals,
as a shared object (test infrastructure only)."""
import ctypes
import os
import subprocess

from paper_2109_12626_gb300 import build as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def load(out_dir: str) -> ctypes.CDLL:
    lib = B.build()
    so = os.path.join(out_dir, "cells_protocol.so")
    r = subprocess.run([B.nvcc(), *B.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                        "-Xcompiler", "-fPIC,-Wall", "-I", B.INCLUDE, "-I", B.CSRC, "-shared",
                        os.path.join(ROOT, "tests", "cells_protocol.cu"), "-o", so,
                        "-cudart", "static", lib, "-Xlinker", "-rpath," + os.path.dirname(lib)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return ctypes.CDLL(so)
