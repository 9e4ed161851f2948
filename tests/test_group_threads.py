"""CPU test of the host threads behind a batch's groups of gates: every part is there when its group's
step runs, and a step that fails or throws ends the threads instead of the process."""
import ctypes
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_steps_see_whole_groups_and_may_fail(tmp_path):
    out = str(tmp_path / "libgroups.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-shared", "-fPIC",
                    os.path.join(ROOT, "tests", "group_threads_harness.cpp"), "-o", out], check=True)
    # in a child: an exception that meets running threads ends the process
    code = f"""
import ctypes
lib = ctypes.CDLL({out!r})
for workers in (1, 2, 7):
    for groups in (1, 3):
        for at in range(groups):
            for how in (0, 1, 2):
                steps = (ctypes.c_int * groups)()
                r = lib.run_groups(workers, groups, at, how, steps)
                assert r == (1 if how == 2 else 0), (workers, groups, at, how, r)
                ran = groups if how == 0 else at + 1
                assert list(steps) == [workers] * ran + [-1] * (groups - ran), list(steps)
print("done")
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "done", r.stderr


def test_small_tables_go_in_one_group(tmp_path):
    out = str(tmp_path / "libgroups.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-shared", "-fPIC",
                    os.path.join(ROOT, "tests", "group_threads_harness.cpp"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    cut = (ctypes.c_long * 4)()

    def cuts(gates, nbytes, one_chunk=1):
        n = lib.group_cuts(ctypes.c_ulong(gates), ctypes.c_ulong(nbytes), one_chunk, cut)
        return list(cut)[:n + 1]
    assert cuts(27, 13 << 10) == [0, 27] and cuts(400, (512 << 10) - 1) == [0, 400]
    assert cuts(7, 1 << 30) == [0, 7] and cuts(24, 1 << 30, 0) == [0, 24]
    for gates in (8, 9, 23, 100):
        c = cuts(gates, 512 << 10)
        assert c[0] == 0 and c[-1] == gates and len(c) == 4 and all(a < b for a, b in zip(c, c[1:]))
