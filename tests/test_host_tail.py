"""The plan of the fused V-cycle tail, built for the host: slabs, shared-memory
arrays, halo writes and cluster barriers of every block, for hierarchies of
powers of two, of other sizes (with a swept coarsest level), of few and of many
planes, with walls and periodic axes, and clusters of 1 to 16 blocks.  No GPU
needed."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1803_00417_gb300", "csrc")


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("tail") / "tail_check")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    os.path.join(HERE, "host", "tail_check.cu"), "-o", exe], check=True, capture_output=True, text=True)
    return exe


@pytest.mark.parametrize("n,per", [((2, 2), "000"), ((64, 64), "000"), ((34, 6), "000"), ((6, 98), "010"),
                                   ((30, 10), "100"), ((128, 48), "110"), ((18, 22), "000"), ((4, 4, 4), "000"),
                                   ((32, 32, 32), "000"), ((36, 28, 20), "000"), ((6, 10, 2), "000"),
                                   ((48, 32, 32), "110"), ((16, 16, 34), "001"), ((14, 14, 14), "111"),
                                   ((2, 2, 70), "000"), ((70, 2, 2), "000")])
def test_tail_plan(harness, n, per):
    r = subprocess.run([harness, str(len(n)), *(str(v) for v in (list(n) + [1])[:3]), per], capture_output=True,
                       text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
