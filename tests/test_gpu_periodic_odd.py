"""Periodic boxes whose coarsest level is swept and has an odd number of cells
along a periodic axis (22 -> 11, 20 -> 10 -> 5): its first and last cells are
neighbours of one colour through the wrap.  In FP64 and mixed precision, with
the fused tail (several slabs along the periodic axis among them) and with the
one-block bottom kernels: two runs give the same bits, and a step agrees with
the oracle.

The oracle's grids keep periodic axes even, so its hierarchy stops above that
level, with more sweeps there: the same equations solved another way.

Tolerances: every solve stops at max|r| <= 1e-10 max|b| on both sides.  The
viscous inverse has norm 1 at most, so u is off by some 2e-10 max|b|, a few
times that against its rms: 1e-9.  The nodal right-hand side is 1e3 at these
sizes and the inverse Laplacian of the unit box below 1/8: 2.5e-8 on a pressure
of order 1: 1e-7."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle.grid import Grid  # noqa: E402
from oracle.multigrid import SolverParams  # noqa: E402
from oracle.step import Rheology, step  # noqa: E402
from paper_1803_00417_gb300.inputs import random_state  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_00417_gb300 import build

    build.build()


def _rel(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b))


@pytest.mark.parametrize("n,per", [((22, 34), "10"), ((22, 34), "01"), ((44, 52), "11"), ((20, 28, 12), "100"),
                                   ((20, 28, 12), "011"), ((12, 20, 36), "001"), ((20, 28, 12), "111")])
def test_odd_periodic_bottom(monkeypatch, n, per):
    from paper_1803_00417_gb300.hbflow import FP64, MIXED, HBFlow

    can = Grid.can_coarsen
    monkeypatch.setattr(Grid, "can_coarsen",
                        lambda s: can(s) and all(s.n[a] % 4 == 0 for a in range(s.d) if s.periodic[a]))
    d, per = len(n), tuple(v == "1" for v in per)
    h = 1.0 / max(n)
    wall = np.zeros((d, 2, d))
    if not per[d - 1]:
        wall[d - 1, 1, 0] = 1.0
    rh = Rheology(K=1.0, n=1.0, tau_y=2.0, m=1e4)
    u, p = random_state(n, seed=sum(n))
    for a in range(d):
        if per[a]:
            p = np.concatenate([np.delete(p, -1, a), np.take(p, [0], a)], a)
    ref = step(Grid(n, h, periodic=per, wall_u=wall), u, p, 0.5 * h, rh, params=SolverParams(nu_bottom=300))
    for precision in (FP64, MIXED):
        for tail in (None, 0):
            bits = []
            for _ in range(2):
                sim = HBFlow(n, h, wall, precision=precision)
                sim.set_periodic(per)
                sim.set_rheology(rh.K, rh.n, rh.tau_y, rh.m, rh.reg_power)
                if tail is not None:
                    sim.set_tail(tail)
                sim.set_velocity(u)
                sim.set_pressure(p)
                st = sim.step(0.5 * h)
                assert all(st[k]["converged"] for k in ("mac", "visc", "nodal")), st
                assert _rel(np.array(sim.velocity()), np.array(ref.u)) < 1e-9
                assert _rel(sim.pressure(), ref.p) < 1e-7
                bits.append(np.concatenate([sim.get_field("U"), sim.get_field("P")]))
                sim.close()
            assert np.array_equal(bits[0], bits[1])
