"""Host decisions of first-use plans, on the CPU: the library's set-up code runs on
fakes of the CUDA runtime calls (tests/host/fake_cuda.h), so that an allocation
can fail, and a stream be under capture, without a GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HOST = os.path.join(ROOT, "tests", "host")
CSRC = os.path.join(ROOT, "paper_1506_07577_gb300", "csrc")


def _run(tmp_path, name, sources, stdin=""):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / name
    flags = ["-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr", "-O1", "-include",
             os.path.join(HOST, "fake_cuda.h"), "--threads", "4"]
    subprocess.run([nvcc, *flags, *[os.path.join(CSRC, s) for s in sources], os.path.join(HOST, name + ".cu"), "-o",
                    str(exe)], check=True, capture_output=True)
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="")   # its pointers are the host's
    r = subprocess.run([str(exe)], input=stdin, env=env, capture_output=True, text=True, timeout=60)
    if r.returncode == 77:
        pytest.skip("a GPU is visible")
    assert r.returncode == 0, r.stderr
    return [tuple(int(x) for x in line.split()) for line in r.stdout.splitlines()]


def test_assembled_stiffness_stays_in_its_storage(tmp_path):
    """(status, on rows, in blocks) per assembly.  Captured products read K where it
    was when they were captured: K assembled into the edge blocks for want of memory
    stays there when there is memory again."""
    got = _run(tmp_path, "assembly_storage", ["edges.cu", "row_matrix.cu"])
    assert got == [(0, 0, 1), (0, 0, 1), (0, 0, 1),   # FP32: no room, room again, captured
                   (1, 0, 0), (0, 1, 0), (0, 1, 0)]   # FP64: first use captured, not captured, captured


def test_element_records_end_with_the_tets(tmp_path):
    """Every size modulo a block of 64: the warps write each record once and none past
    the last, also where a block's second warp has no tet."""
    sizes = list(range(1, 200)) + [1551, 1310720, 1310721]
    got = _run(tmp_path, "warp_tets", [], "".join(f"{n} 64\n" for n in sizes))
    assert got == [(n, n) for n in sizes]


def test_batch_scratch_after_host_memory_ran_out(tmp_path):
    """(first call failed, second call's tables whole), the first call's k-th host
    allocation failing: a half-built scratch is not taken for a finished one."""
    got = _run(tmp_path, "batch_scratch", [])
    assert len(got) > 5 and got[-1] == (0, 1)
    assert all(g == (1, 1) for g in got[:-1]), got
