"""The branch-free homogeneous-wall viscous sweep and residual of the V-cycles'
levels with stored face viscosities, built for the host, against the general
forms on every cell (walls, periodic axes, two cells per axis; FP64 and FP32;
beta / h^2 from negligible to dominant).  The bound is rounding (see the
harness).  No GPU needed."""

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
    exe = str(tmp_path_factory.mktemp("hom") / "hom_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", CSRC, os.path.join(HERE, "host", "hom_check.cu"), "-o", exe],
                   check=True, capture_output=True, text=True)
    return exe


@pytest.mark.parametrize("n,per", [((2, 2), "000"), ((5, 3), "000"), ((8, 6), "100"), ((2, 4), "110"),
                                   ((2, 2, 2), "000"), ((3, 5, 2), "000"), ((9, 7, 5), "000"), ((4, 6, 8), "100"),
                                   ((4, 2, 6), "010"), ((6, 4, 2), "001"), ((2, 4, 2), "111")])
@pytest.mark.parametrize("beta", [1e-6, 1e-2, 10.0])
def test_homogeneous_forms_match_the_general_ones(harness, n, per, beta):
    args = [str(len(n)), *(str(v) for v in (list(n) + [1])[:3]), per, str(beta), str(17 + sum(n))]
    r = subprocess.run([harness, *args], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
