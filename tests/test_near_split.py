"""CPU test of the digit split's short cut for components near their row's largest exponent: the
same words as the general form for every spread it accepts (0 to 31)."""
import ctypes
import os
import subprocess

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_near_split_equals_general_form(tmp_path):
    out = str(tmp_path / "libnear.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC",
                    os.path.join(ROOT, "tests", "near_split_harness.cpp"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    lib.near_split_mismatches.restype = ctypes.c_long
    rng = np.random.default_rng(5)
    n = 1 << 18
    mant = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    mant[::4] &= ~((np.uint64(1) << rng.integers(0, 52, n // 4).astype(np.uint64)) - np.uint64(1))
    mant[1::4] |= (np.uint64(1) << rng.integers(0, 52, n // 4).astype(np.uint64)) - np.uint64(1)
    spread = rng.integers(0, 32, n).astype(np.uint32)
    ef = rng.integers(1, 2047 - spread.astype(np.int64), n).astype(np.uint64)
    ef[:64] = 1
    sign = rng.integers(0, 2, n, dtype=np.uint64) << np.uint64(63)
    x = (sign | ef << np.uint64(52) | mant).view(np.float64)
    assert lib.near_split_mismatches(x.ctypes.data_as(ctypes.c_void_p), spread.ctypes.data_as(ctypes.c_void_p),
                                     ctypes.c_long(n)) == 0
