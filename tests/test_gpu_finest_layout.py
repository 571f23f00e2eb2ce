"""Which layout the mixed viscous solve keeps its FP32 finest level in: the
library's rule (stored faces up to 2^19 cells, above them colour-split where
the grid can have it), and the two that a caller can ask for on any grid
(hbf_set_split_layout); the colour-split kernels on both sides of 2^19 cells,
with a half row of even and of odd length, against the natural layout, with the
previous-increment guess and across changes of layout, and with a network's
direction (whose residual is restricted from the split layout).

Tolerance: as the layouts' test, 1e-8 of the largest value (every solve stops
at 1e-10; the layouts differ in the summation order of the dot products)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1803_00417_gb300.inputs import cavity, random_state  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_00417_gb300 import build

    build.build()


@pytest.mark.parametrize("n,per,rule,asked", [
    ((30, 18, 22), "000", "stored faces", "colour-split"), ((80, 80, 80), "000", "stored faces", "colour-split"),
    ((128, 64, 64), "000", "stored faces", "colour-split"), ((128, 64, 66), "000", "colour-split", "colour-split"),
    ((81, 82, 82), "000", "natural", "natural"), ((96, 96, 96), "100", "natural", "natural"),
    ((64, 64, 64), "001", "stored faces", "natural"), ((512, 512), "000", "stored faces", "natural"),
    ((1024, 640), "000", "natural", "natural")])
def test_layout_in_use(n, per, rule, asked):
    from paper_1803_00417_gb300.hbflow import FP64, MIXED, HBFlow, HBFlowError

    sim = HBFlow(n, 1.0 / max(n), precision=MIXED)
    if "1" in per:
        sim.set_periodic([v == "1" for v in per])
    assert sim.finest_layout() == rule
    sim.set_split_layout(1)
    assert sim.finest_layout() == asked
    sim.set_fused_sweep(1)
    assert sim.finest_layout() == "natural"
    sim.set_fused_sweep(0)
    sim.set_split_layout(0)
    assert sim.finest_layout() == "natural"
    sim.close()
    sim = HBFlow((8, 8), 0.125, precision=FP64)
    with pytest.raises(HBFlowError):
        sim.finest_layout()
    sim.close()


def _run(n, layouts, guess=0, net=None):
    from paper_1803_00417_gb300.hbflow import MIXED, HBFlow, set_visc_guess_model

    cfg = cavity(n, Re=100.0, Bi=10.0, Pa=1e5, nexp=1.5)
    u, p = random_state(cfg["n"], seed=sum(n))
    sim = HBFlow(cfg["n"], cfg["h"], cfg["wall_u"], precision=MIXED)
    sim.set_rheology(cfg["K"], cfg["nexp"], cfg["tau_y"], cfg["m"])
    if guess:
        sim.set_visc_guess(guess)
    if net:
        set_visc_guess_model(sim, net, 1)
    sim.set_velocity(u)
    sim.set_pressure(p)
    for on in layouts:
        if on is not None:
            sim.set_split_layout(on)
            assert sim.finest_layout() == ("colour-split" if on else "natural")
        st = sim.step(cfg["dt"])
        for k in ("mac", "visc", "nodal"):
            assert st[k]["converged"], (k, st[k])
    out = np.concatenate([sim.get_field("U"), sim.get_field("P")])
    sim.close()
    return out


# half rows of 15, 12 and 64 cells; the last one above the rule's limit
@pytest.mark.parametrize("n", [(30, 18, 22), (24, 40, 12), (128, 96, 64)])
@pytest.mark.parametrize("guess", [0, 1])
def test_split_against_natural(n, guess):
    nat = _run(n, [0, 0, 0], guess)
    for layouts in ([1, 1, 1], [None, None, None], [None, 1, 1], [1, 0, 1]):
        assert np.max(np.abs(_run(n, layouts, guess) - nat)) <= 1e-8 * np.max(np.abs(nat)), layouts


def test_network_direction_from_the_split_layout():
    from paper_1803_00417_gb300.hbflow import UNet
    from paper_1803_00417_gb300.learned import cell_box

    n = (48, 32, 16)
    net = UNet(cell_box((24, 16, 8)), seed=3)
    nat = _run(n, [0, 0], 2, net)
    for layouts in ([1, 1], [None, None]):
        assert np.max(np.abs(_run(n, layouts, 2, net) - nat)) <= 1e-8 * np.max(np.abs(nat))
    net.close()
