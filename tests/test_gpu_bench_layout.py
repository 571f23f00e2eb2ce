"""What bench.py reports of the FP32 finest level is what the library runs, on
both sides of the size where its choice changes and in FP64."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import bench  # noqa: E402


@pytest.mark.parametrize("n,precision,want", [((64, 64, 64), 1, "stored faces"), ((96, 96, 96), 1, "colour-split"),
                                              ((64, 64, 64), 0, None)])
def test_reported_layout(n, precision, want):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_00417_gb300 import build

    build.build()
    from paper_1803_00417_gb300.hbflow import HBFlow

    sim = HBFlow(n, 1.0 / n[0], precision=precision)
    assert bench.finest_layout(sim, precision) == want
    sim.close()
