"""The host-side launch rules (csrc headers), compiled into a library of their own."""
import collections
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
    lib.shared_part_rows.restype = ctypes.c_int64
    lib.shared_part_rows.argtypes = [ctypes.c_int64, ctypes.c_int32, ctypes.c_int32]
    lib.decode_shape.restype = None
    lib.decode_shape.argtypes = [ctypes.c_int32] * 6 + [ctypes.c_int64] + [ctypes.c_int32] * 2 + \
        [ctypes.POINTER(ctypes.c_int32)]
    return lib


Shape = collections.namedtuple("Shape", "sub per_sm pace merge_max one_split by_length wide combine")


def splits_of(tokens: int) -> int:
    """Splits of a table of so many tokens (the bound that sizes the workspace)."""
    tiles = -(-tokens // 16)
    return max(-(-tiles // 128), min(16, -(-tiles // 64)))


def pool_part_rows(max_batch, max_context, hq, hkv, sms) -> int:
    """Rows for partials that a pool allocates."""
    return rules().shared_part_rows(max_batch * hq * splits_of(max_context), sms, hq // hkv)


def decode_shape(tokens, batch, *, bt=16, hq=32, hkv=4, layers=1, part_rows=1 << 40, sms=152,
                 overlap=False) -> Shape:
    """The launch shape of a call over tables of `tokens` tokens (rounded up to blocks)."""
    out = (ctypes.c_int32 * 8)()
    rules().decode_shape(-(-tokens // bt), bt, hq, hkv, layers, batch, part_rows, sms, overlap, out)
    return Shape(*out)
