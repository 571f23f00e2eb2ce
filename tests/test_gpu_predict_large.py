"""The predictor on 3D boxes that its marching kernels take by their rules
(walls and periodic axes) against the oracle's face states: slopes alone on
boxes that leave the tiles of the transverse terms half empty (an x extent of
one cell more than a block of the slopes along x, of three quarters of a tile),
and both on boxes whose x, y and z extents are no multiple of the tiles and the
chunks, of few planes and of many chunks.

Tolerance: the states are u plus products of a few rounded terms with the
slopes (1e-12 relative L2, as on the small grids)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle.godunov import face_states  # noqa: E402
from oracle.grid import Grid, nodes_unique  # noqa: E402
from oracle.operators import cell_grad_nodal  # noqa: E402
from paper_1803_00417_gb300.inputs import cavity, random_state  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_00417_gb300 import build

    build.build()


@pytest.mark.parametrize("n,per", [((60, 60, 60), "000"), ((129, 48, 40), "000"), ((48, 80, 60), "110"),
                                   ((120, 60, 60), "000"), ((127, 62, 66), "000"), ((64, 12, 1000), "000"),
                                   ((64, 600, 13), "000"), ((64, 96, 64), "101"), ((120, 60, 60), "010"),
                                   ((128, 64, 64), "111")])
def test_predictor_matches_oracle(n, per):
    from paper_1803_00417_gb300.hbflow import HBFlow

    per = tuple(v == "1" for v in per)
    cfg = cavity(n, Re=10.0, Bi=0.1, Pa=100.0, nexp=0.8)
    rng = np.random.default_rng(sum(n))
    walls = rng.uniform(-1.0, 1.0, size=(3, 2, 3))
    for a in range(3):
        walls[a, :, a] = 0.0
        if per[a]:
            walls[a] = 0.0
    u, p = random_state(n, seed=sum(n))
    for a in range(3):
        if per[a]:
            p = np.concatenate([np.delete(p, -1, a), np.take(p, [0], a)], a)
    sim = HBFlow(n, cfg["h"], walls)
    if any(per):
        sim.set_periodic(per)
    sim.set_rheology(cfg["K"], cfg["nexp"], cfg["tau_y"], cfg["m"])
    sim.set_velocity(u)
    sim.set_pressure(p)
    sim.compute_viscosity()
    sim.predict(cfg["dt"])
    g = Grid(n, cfg["h"], periodic=per, wall_u=walls)
    F = [-v for v in cell_grad_nodal(nodes_unique(p, g), g)]
    for name, ref in zip(("UL", "UR"), face_states(u, F, g, cfg["dt"])):
        got = sim.face_field(name, 3)
        for a in range(3):
            x, y = np.array(got[a]), np.array(ref[a])
            assert np.linalg.norm(x - y) <= 1e-12 * np.linalg.norm(y)
            assert np.max(np.abs(x - y)) <= 1e-11 * np.max(np.abs(y))
    sim.close()
