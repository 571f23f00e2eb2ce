"""Mixed precision on boxes with periodic axes: the FP32 forms with wraps (the
V-cycle tail with its halo stores through the wrap, the sweeps, residual and
operator with stored faces, and above 2^19 cells the sweeps with the cell
viscosity) against the oracle, and the default route against the same solves
level by level and in the natural layout, cycle counts among them (a wrong wrap
in a preconditioner costs iterations, not the result).  The slowest axis is
periodic and cut into several slabs in some.

Tolerances: 1e-6 against the oracle in the velocity and ten times that in the
pressure, as the mixed steps with walls; 1e-8 of the largest value between the
routes; and their cycles within a quarter, and one, of each other (they round
differently, so a solve may stop a cycle earlier or later)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle.grid import Grid  # noqa: E402
from oracle.step import Rheology, step  # noqa: E402
from paper_1803_00417_gb300.inputs import random_state  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_00417_gb300 import build

    build.build()


def _case(n, per, seed):
    d, per = len(n), tuple(v == "1" for v in per)
    h = 1.0 / max(n)
    wall = np.zeros((d, 2, d))
    if not per[d - 1]:
        wall[d - 1, 1, 0] = 1.0
    u, p = random_state(n, seed=seed)
    for a in range(d):
        if per[a]:
            p = np.concatenate([np.delete(p, -1, a), np.take(p, [0], a)], a)
    return per, h, wall, Rheology(K=0.1, n=0.8, tau_y=0.2, m=1e4), u, p


def _sim(n, case):
    from paper_1803_00417_gb300.hbflow import MIXED, HBFlow

    per, h, wall, rh, u, p = case
    sim = HBFlow(n, h, wall, precision=MIXED)
    sim.set_periodic(per)
    sim.set_rheology(rh.K, rh.n, rh.tau_y, rh.m, rh.reg_power)
    sim.set_velocity(u)
    sim.set_pressure(p)
    return sim


def _rel(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b))


@pytest.mark.parametrize("n,per", [((32, 24), "10"), ((64, 64), "01"), ((32, 64), "11"), ((16, 12, 10), "110"),
                                   ((24, 16, 32), "001"), ((16, 16, 32), "111"), ((32, 32, 16), "010")])
def test_mixed_periodic_step_matches_oracle(n, per):
    case = _case(n, per, sum(n))
    per, h, wall, rh, u, p = case
    sim = _sim(n, case)
    ref = None
    for _ in range(2):
        ref = step(Grid(n, h, periodic=per, wall_u=wall), u if ref is None else ref.u, p if ref is None else ref.p,
                   0.5 * h, rh)
        st = sim.step(0.5 * h)
        for k in ("mac", "visc", "nodal"):
            assert st[k]["converged"] and st[k]["rnorm"] <= 1e-10 * st[k]["bnorm"], (k, st[k])
    assert _rel(np.array(sim.velocity()), np.array(ref.u)) < 1e-6
    assert _rel(sim.pressure(), ref.p) < 1e-5
    sim.close()


# tails from the finest level and below it, stored faces up to 2^19 cells (128 x 64 x 64) and the cell viscosity above
@pytest.mark.parametrize("n,per", [((128, 128), "10"), ((256, 128), "01"), ((512, 512), "11"), ((768, 768), "10"),
                                   ((32, 32, 32), "001"), ((48, 32, 64), "110"), ((64, 64, 96), "111"),
                                   ((128, 64, 64), "100"), ((128, 96, 64), "010")])
def test_mixed_periodic_routes_agree(n, per):
    case = _case(n, per, sum(n))
    outs, cycles = [], []
    for tail, split in ((None, None), (0, None), (None, 0)):
        sim = _sim(n, case)
        if tail is not None:
            sim.set_tail(tail)
        if split is not None:
            sim.set_split_layout(split)
        cyc = []
        for _ in range(2):
            st = sim.step(0.5 * case[1])
            for k in ("mac", "visc", "nodal"):
                assert st[k]["converged"], (k, st[k])
            cyc += [st[k]["cycles"] for k in ("mac", "visc", "nodal")]
        outs.append(np.concatenate([sim.get_field("U"), sim.get_field("P")]))
        cycles.append(cyc)
        sim.close()
    for o, c in zip(outs[1:], cycles[1:]):
        assert np.max(np.abs(o - outs[0])) <= 1e-8 * np.max(np.abs(outs[0]))
        assert all(abs(a - b) <= 1 + max(a, b) // 4 for a, b in zip(c, cycles[0])), cycles
