"""Calls into single kernels of the library from tests: a translation unit of csrc/ is compiled with a small
C entry into a shared library of its own (what libxbar.so exports is only its C ABI)."""
from __future__ import annotations

import ctypes
import os
import subprocess

from paper_2410_19993_gb300 import build


def compile_probe(folder, name: str, source: str) -> ctypes.CDLL:
    cu, so = os.path.join(str(folder), name + ".cu"), os.path.join(str(folder), name + ".so")
    with open(cu, "w") as f:
        f.write(source)
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-shared", "-o", so, cu],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


def ptr(a) -> ctypes.c_void_p:
    return ctypes.c_void_p(a.data_ptr() if hasattr(a, "data_ptr") else a.ctypes.data)
