"""Builds kernel_units.cu, which exports functions of the kernels' headers one
at a time, and loads it."""
import atexit
import ctypes
import functools
import os
import shutil
import subprocess
import tempfile

from paper_2508_13705_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@functools.lru_cache(maxsize=None)
def lib():
    d = tempfile.mkdtemp(prefix="cgks_units_")
    atexit.register(shutil.rmtree, d, ignore_errors=True)
    so = os.path.join(d, "libunits.so")
    subprocess.run([build._nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.SRC,
                    os.path.join(HERE, "kernel_units.cu"), "-o", so], check=True, capture_output=True, text=True)
    L = ctypes.CDLL(so)
    L.unit_fr_nrow.restype = ctypes.c_longlong
    return L
