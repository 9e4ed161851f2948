"""CPU test of the kernels' one-time setup: once for every device that a process uses, not once for
the first; and no kernel's setup goes round it."""
import ctypes
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_setup_runs_once_per_device(tmp_path):
    out = str(tmp_path / "libdev.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-shared", "-fPIC",
                    os.path.join(ROOT, "tests", "per_device_harness.cpp"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    calls = (ctypes.c_int * 8)()
    assert lib.per_device_calls(8, 6, calls) == 0
    assert list(calls) == [1] * 8


def test_no_function_attribute_is_set_once_per_process():
    for path in glob.glob(os.path.join(ROOT, "paper_2604_03816_gb300", "csrc", "*.cu")):
        text = open(path).read()
        for m in re.finditer(r"cudaFuncSetAttribute\(|cudaOccupancyMaxActiveClusters\(", text):
            before = text[:m.start()]
            assert before.rfind("PerDevice") > before.rfind("call_once"), (os.path.basename(path), m.start())
