"""The order of a coarsest level's sweeps, built for the host: on walls and on
periodic axes of even and odd cell counts (a periodic 40 coarsens to 5 cells,
whose first and last have one colour and are neighbours through the wrap) every
sweep visits every point once, and no two points of one pass are neighbours; for
the one-block kernels and for both forms of the fused tail (whose slot form
stores a pass's values behind a barrier on such levels and may hold the
neighbours that the wrap makes).  No GPU needed."""

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
    exe = str(tmp_path_factory.mktemp("order") / "order_check")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    os.path.join(HERE, "host", "order_check.cu"), "-o", exe], check=True, capture_output=True, text=True)
    return exe


_SIZES = [(3, 2), (3, 5), (11, 17), (6, 9), (4, 4), (3, 4, 5), (5, 7, 9), (5, 6, 8), (9, 3, 4), (6, 4, 7), (3, 3, 3),
          (4, 6, 2)]
_CASES = [(n, f"{q:03b}"[::-1]) for n in _SIZES for q in range(1 << len(n))]


@pytest.mark.parametrize("n,per", _CASES)
def test_no_pass_updates_two_neighbours(harness, n, per):
    r = subprocess.run([harness, str(len(n)), *(str(v) for v in (list(n) + [1])[:3]), per], capture_output=True,
                       text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
