"""Multigrid solves at the sizes where their paths change: grids that are their
own coarsest level, with exact (at most 128 unknowns) and swept bottoms; small
FP32 finest levels with stored faces that run wholly inside the V-cycle tail,
against the same solves level by level and in the general layout; the first
grids above that range; and a batch's tails likewise.

Tolerances: the oracle's steps to 1e-10 (each side stops its solves at 1e-10 of
the right-hand side and the steps scale that down); solver routes of the mixed
precision against each other to 1e-8, as the layouts' test."""

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


# 80^3 is the last cube whose finest level stores its faces; the grids with more cells end inside
# the operator's 64-cell tile (48, 112 and 160 cells along x) and at its edge (128)
@pytest.mark.parametrize("n", [(24, 20, 12), (12, 40, 28), (80, 80, 80), (112, 80, 64), (48, 128, 96), (160, 64, 56),
                               (128, 64, 80), (72, 48)])
def test_mixed_routes_agree(n):
    cfg = cavity(n, Re=100.0, Bi=10.0, Pa=1e4, nexp=1.2)
    u, p = random_state(cfg["n"], seed=sum(n))
    outs = []
    for tail, split in ((None, None), (0, None), (None, 0)):
        sim = _sim(cfg, u, p, 1)
        if tail is not None:
            sim.set_tail(tail)
        if split is not None:
            sim.set_split_layout(split)
        for _ in range(2):
            st = sim.step(cfg["dt"])
            for k in ("mac", "visc", "nodal"):
                assert st[k]["converged"], (k, st[k])
                assert st[k]["rnorm"] <= 1e-10 * st[k]["bnorm"]
        outs.append(np.concatenate([sim.get_field("U"), sim.get_field("P")]))
        sim.close()
    for other in outs[1:]:
        assert np.max(np.abs(other - outs[0])) <= 1e-8 * np.max(np.abs(outs[0]))


# the last level sizes that a batch's default tail takes in mixed precision, and the first above
@pytest.mark.parametrize("sizes", [((128, 128), (96, 64)), ((160, 128), (64, 64), (256, 256))])
def test_batch_default_tail_matches_level_by_level(sizes):
    from paper_1803_00417_gb300.hbflow import MIXED, Batch

    cfgs = [cavity(n, Re=100.0, Bi=10.0, Pa=1e4, nexp=1.2) for n in sizes]
    outs = []
    for tail in (None, 0):
        B = Batch([c["n"] for c in cfgs], [c["h"] for c in cfgs], [c["wall_u"] for c in cfgs], precision=MIXED)
        if tail is not None:
            B.set_tail(tail)
        for i, c in enumerate(cfgs):
            v = B.cavity(i)
            v.set_rheology(c["K"], c["nexp"], c["tau_y"], c["m"])
            u, p = random_state(c["n"], seed=sum(c["n"]))
            v.set_velocity(u)
            v.set_pressure(p)
        B.set_dt([c["dt"] for c in cfgs])
        for _ in range(2):
            st = B.step()
            assert all(s[k]["converged"] for s in st for k in ("mac", "visc", "nodal")), st
        outs.append([np.concatenate([B.cavity(i).get_field("U"), B.cavity(i).get_field("P")])
                     for i in range(len(cfgs))])
        B.close()
    for a, b in zip(*outs):
        assert np.max(np.abs(b - a)) <= 1e-8 * np.max(np.abs(a))
