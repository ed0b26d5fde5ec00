"""The host-side launch rules (csrc headers), compiled into a library of their own."""
import ctypes
import functools
import os
import shutil
import subprocess
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2609_25782_gb300", "csrc")


@functools.cache
def rules() -> ctypes.CDLL:
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    with tempfile.TemporaryDirectory() as d:
        so = os.path.join(d, "launch_rules.so")
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-I", cuda,
                        os.path.join(HERE, "launch_rules.cpp"), "-o", so], check=True)
        lib = ctypes.CDLL(so)
    for name in ("grid_ctas", "copy_threads", "inline_blocks"):
        getattr(lib, name).restype = ctypes.c_int64
    lib.grid_ctas.argtypes = [ctypes.c_int64, ctypes.c_int64]
    return lib
