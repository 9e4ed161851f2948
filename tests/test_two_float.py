"""CPU test of the expectations' running sums: over runs as long as a thread's at 34 qubits their
error stays so small that a block's sum of 4096 of them is exact to FP64's rounding."""
import ctypes
import math
import os
import subprocess

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_long_runs_keep_their_accuracy(tmp_path):
    out = str(tmp_path / "libtwo.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC",
                    os.path.join(ROOT, "tests", "two_float_harness.cpp"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    lib.two_float_sum.restype = ctypes.c_double
    rng = np.random.default_rng(0)
    for n in (1, 127, 128, 129, 1000, 2200, 14000):
        for signed in (False, True):
            mine = []
            for _ in range(40):
                x = rng.exponential(size=n).astype(np.float32)
                if signed:
                    x *= rng.choice([-1, 1], n).astype(np.float32)
                got = lib.two_float_sum(x.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(n))
                size = float(np.sum(np.abs(x), dtype=np.float64))
                mine.append((got - math.fsum(x.astype(np.float64))) / size)
            # 2^-49 / sqrt(4096) = 2^-55 of a block's total
            assert np.sqrt(np.mean(np.square(mine))) <= 2.0 ** -49, (n, signed)
