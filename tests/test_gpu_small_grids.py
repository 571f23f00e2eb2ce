"""Multigrid solves on grids that are their own coarsest level, with exact (at
most 128 unknowns) and swept bottoms, against the oracle.

Tolerance: the oracle's steps to 1e-10 (each side stops its solves at 1e-10 of
the right-hand side and the steps scale that down)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle.grid import Grid  # noqa: E402
from oracle.step import Rheology, step  # noqa: E402
from paper_1803_00417_gb300.inputs import cavity, random_state  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_00417_gb300 import build

    build.build()


def _sim(cfg, u, p, precision):
    from paper_1803_00417_gb300.hbflow import HBFlow

    sim = HBFlow(cfg["n"], cfg["h"], cfg["wall_u"], precision=precision)
    sim.set_rheology(cfg["K"], cfg["nexp"], cfg["tau_y"], cfg["m"])
    sim.set_velocity(u)
    sim.set_pressure(p)
    return sim


# viscous unknowns 24 (exact) to 375 (swept), cells 12 to 125, nodes 20 to 216
@pytest.mark.parametrize("n", [(4, 3), (5, 7), (7, 9), (8, 8), (11, 5), (3, 5, 3), (5, 5, 5), (4, 4, 4), (6, 10, 4)])
def test_coarsest_grids_match_oracle(n):
    cfg = cavity(n, Re=10.0, Bi=1.0, Pa=100.0, nexp=0.8)
    u, p = random_state(cfg["n"], seed=sum(n))
    sim = _sim(cfg, u, p, 0)
    ref = step(Grid(cfg["n"], cfg["h"], wall_u=cfg["wall_u"]), u, p, cfg["dt"],
               Rheology(cfg["K"], cfg["nexp"], cfg["tau_y"], cfg["m"]))
    st = sim.step(cfg["dt"])
    assert all(st[k]["converged"] for k in ("mac", "visc", "nodal")), st
    got, want = np.array(sim.velocity()), np.array(ref.u)
    assert np.linalg.norm(got - want) <= 1e-10 * np.linalg.norm(want)
    sim.close()
