"""CPU test of the choice between tiled reads of many Z strings and the kernels with a weight per
string and amplitude: unlike strings must not cost a read per three of them, chains stay tiled."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("split") / "libsplit.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC",
                    os.path.join(ROOT, "tests", "z_split_harness.cpp"), "-o", out], check=True)
    lib = ctypes.CDLL(out)

    def call(z, n, dtype, states=1, batch=False):
        z = np.asarray(z, dtype=np.uint64)
        g = np.zeros(z.size, dtype=np.int8)
        lib.split_z(z.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(z.size), min(n, 12 - dtype),
                    ctypes.c_double(float(states) * 2.0 ** n), int(batch), dtype, g.ctypes.data_as(ctypes.c_void_p))
        return g.astype(bool)
    return call


def _unlike(n, m):
    """m strings with a bit in the tile and no two high parts alike."""
    return [1 | ((i + 1) << 12) for i in range(m)]


def test_unlike_strings_go_to_the_general_kernels(split):
    for n in (24, 26, 30):
        assert split(_unlike(n, 32), n, 1).all()                     # 11 tiled reads against one
        assert split(_unlike(n, 96), n, 1).all()
        assert not split(_unlike(n, 96), n, 0).any()                 # FP64 weights against FP32 sums
        assert not split(_unlike(n, 3), n, 1).any()                  # one tiled read
    assert split(_unlike(20, 32), 20, 0).all()                       # launches count there
    assert split(_unlike(18, 32), 18, 0, 96, True).all() and split(_unlike(18, 32), 18, 1, 96, True).all()


def test_chains_and_pairs_stay_tiled(split):
    for n in (20, 24, 28):
        chain = [3 << i for i in range(n - 1)]
        pairs = [1 << i | 1 << j for i in range(n) for j in range(i)]
        for dtype in (0, 1):
            assert not split(chain, n, dtype).any() and not split(pairs, n, dtype).any()
    assert not split([3 << i for i in range(17)], 18, 0, 96, True).any()


def test_a_few_unlike_strings_beside_a_chain(split):
    n = 26
    g = split([3 << i for i in range(n - 1)] + _unlike(n, 40)[8:], n, 1)
    assert not g[:n - 1].any() and g[n - 1:].sum() >= 30             # the chain's read takes at most two along
    g = split([3 << i for i in range(n - 1)] + [1 | 5 << 14, 1 | 7 << 20], n, 1)
    assert not g.any()
