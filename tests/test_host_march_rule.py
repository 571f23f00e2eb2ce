"""Which boxes the predictor's marching kernels and the marching nodal residual
take, built for the host: each side of the rules as it was measured (faster or
slower than one thread per cell or node, GB300); and which launches of the
explicit stages start while their predecessor drains.  No GPU needed."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1803_00417_gb300", "csrc")

SRC = """
#include <cstdlib>
#include <cstring>
#include "hb_internal.h"
#include "hb_explicit_march.cuh"
#include "hb_mg_kernels.cuh"
int main(int argc, char** argv) {
  if (argc == 2) return hb::stage_early(std::atoi(argv[1])) ? 11 : 10;
  hb::Geom g;
  std::memset(&g, 0, sizeof g);
  g.ncell = g.nnode = 1;
  for (int a = 0; a < 3; ++a) {
    g.ncell *= g.n[a] = std::atoi(argv[1 + a]);
    g.nnode *= g.n[a] + 1;
  }
  return 10 + (hb::slopes_march(g) ? 1 : 0) + (hb::hats_march(g) ? 2 : 0) + (hb::nodal_march_level(g) ? 4 : 0);
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("march")
    (d / "rule.cu").write_text(SRC)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr", "-I",
                    CSRC, str(d / "rule.cu"), "-o", str(d / "rule")], check=True, capture_output=True, text=True)
    return str(d / "rule")


# (slopes, transverse terms, nodal residual) by march
@pytest.mark.parametrize("n,want", [
    ((40, 40, 40), (0, 0, 0)), ((48, 48, 48), (0, 0, 0)), ((72, 56, 40), (0, 0, 0)), ((56, 56, 56), (0, 0, 0)),
    ((47, 500, 500), (0, 0, 1)), ((60, 60, 60), (1, 0, 1)), ((66, 64, 64), (1, 0, 1)), ((80, 80, 80), (1, 0, 1)),
    ((96, 64, 64), (1, 0, 1)), ((130, 60, 60), (1, 0, 1)), ((64, 96, 64), (1, 1, 1)), ((120, 60, 60), (1, 1, 1)),
    ((128, 64, 64), (1, 1, 1)), ((128, 128, 128), (1, 1, 1)), ((256, 256, 256), (1, 1, 1)),
    ((64, 70000, 6), (0, 0, 0)), ((128, 64, 16), (0, 0, 0)), ((128, 96, 16), (0, 0, 1)), ((64, 64, 48), (0, 0, 1)),
    ((256, 512, 15), (1, 1, 0))])
def test_rule(harness, n, want):
    r = subprocess.run([harness, *map(str, n)], capture_output=True, timeout=60)
    assert r.returncode - 10 == want[0] + 2 * want[1] + 4 * want[2]


# blocks of 256 cells of the cubes 26, 28, 32, 36, 40, 48, 53, 54 and 128
@pytest.mark.parametrize("blocks,early", [(69, 1), (86, 0), (128, 0), (183, 1), (250, 0), (432, 0), (582, 0), (616, 1),
                                          (2432, 1)])
def test_early_start(harness, blocks, early):
    assert subprocess.run([harness, str(blocks)], timeout=60).returncode - 10 == early
