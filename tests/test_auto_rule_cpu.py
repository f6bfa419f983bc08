"""EBB_REDUCE_AUTO of FP64 maps, on the CPU: three threads per tet on few tets, one with
atomics on more, and the tiles' own sums where so many tets meet in one vertex that
its atomics would be the map's time."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
ATOMIC, TILED, COOP = 0, 3, 6   # include/ebb.h


def test_auto_reduction_of_fp64_maps(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "auto_rule"
    subprocess.run([nvcc, "-std=c++17", "-O1", os.path.join(ROOT, "tests", "host", "auto_rule.cu"), "-o", str(exe)],
                   check=True, capture_output=True)
    cases = {(0, 0): COOP, (8191, 24): COOP, (8191, 2560): COOP, (8191, 2561): TILED, (8192, 24): ATOMIC,
             (8192, 2560): ATOMIC, (8192, 2561): TILED, (1 << 33, 24): ATOMIC, (20000, 20000): TILED}
    out = subprocess.run([str(exe)], input="".join(f"{t} {m}\n" for t, m in cases), capture_output=True, text=True,
                         check=True).stdout.split()
    assert [int(x) for x in out] == list(cases.values())
