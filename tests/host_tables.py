"""The stream and set kernels' tables as the host compiler lays them out, read from a compiled program
(tests/native/host_tables.cpp, built on first use; no GPU needed)."""
import ctypes
import os
import subprocess
import tempfile

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KEEP = 0x8000                                  # kLeafBit of an edge
RUNS = 16                                      # kSetRuns
FIELD, PAIR, SINGLE = 1, 2, 3                  # stream.kind
_LIB = None


def _lib():
    global _LIB
    if _LIB is None:
        from paper_2412_14975_gb300 import build_lib
        cuda, _ = build_lib._cuda_home()
        tmp = tempfile.TemporaryDirectory()
        out = os.path.join(tmp.name, "host_tables.so")
        subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", build_lib.INC, "-I", build_lib.CSRC,
                               "-I", os.path.join(cuda, "include"), os.path.join(ROOT, "tests", "native", "host_tables.cpp"), "-o", out])
        lib = ctypes.CDLL(out)
        lib.ht_table.restype = ctypes.c_void_p
        lib.ht_table.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_char_p, ctypes.POINTER(ctypes.c_uint64)]
        lib.ht_number.restype = ctypes.c_int64
        lib.ht_number.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_char_p]
        _LIB = lib
    return _LIB


def number(prog, name, dfa=False):
    v = _lib().ht_number(prog, int(dfa), name.encode())
    assert v >= 0, name
    return v


def table(prog, name, dtype, dfa=False):
    size = ctypes.c_uint64(0)
    at = _lib().ht_table(prog, int(dfa), name.encode(), ctypes.byref(size))
    if not at or not size.value:
        return np.zeros(0, dtype=dtype)
    return np.frombuffer(ctypes.string_at(at, size.value), dtype=dtype)
