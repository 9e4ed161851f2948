"""CPU test of the small-state kernel's size rule: whatever cluster the device schedules, a state it
takes gives no thread more than one amplitude."""
import ctypes
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_thread_owns_two_amplitudes(tmp_path):
    out = str(tmp_path / "libfit.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC",
                    os.path.join(ROOT, "tests", "small_fit_harness.cpp"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    for max_c in range(5):
        for n in range(1, 20):
            c = lib.cluster_log2(n, max_c)
            assert c <= max_c and c < n
            if lib.state_fits(n, max_c):
                assert n <= 12 and (1 << n) >> c <= lib.threads(), (n, max_c)
            else:
                assert n > 12 or (1 << n) >> c > lib.threads()
    assert all(lib.state_fits(n, 4) for n in range(1, 13))         # clusters of 16: up to 12 qubits
    assert lib.state_fits(11, 3) and not lib.state_fits(12, 3)     # clusters of 8: up to 11
