"""The 3D FP64 nodal residual that marches along z, on both sides of its limit
of 2e5 nodes (walls and periodic axes), through the residual of a projection
evaluated by the oracle.  The columns are no multiple of a block, the z extents
multiples of the chunk and not.

Tolerance: the solve stops at max|r| <= 1e-10 max|b| with the weighted mean of
the right-hand side removed; the oracle's own rounding adds less than 1e-12."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle.grid import Grid, node_weights, nodes_unique  # noqa: E402
from oracle.operators import cell_grad_nodal, nodal_div, nodal_lap  # noqa: E402
from paper_1803_00417_gb300.inputs import cavity, random_state  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_00417_gb300 import build

    build.build()


@pytest.mark.parametrize("n,per", [((56, 56, 60), "000"), ((64, 64, 48), "000"), ((72, 80, 40), "000"),
                                   ((128, 96, 16), "100"), ((64, 64, 52), "011"), ((48, 64, 64), "111")])
def test_projection_matches_oracle(n, per):
    from paper_1803_00417_gb300.hbflow import HBFlow, from_device_layout, to_device_layout

    per = tuple(v == "1" for v in per)
    cfg = cavity(n, Re=10.0, Bi=0.1, Pa=100.0, nexp=0.8)
    us, p = random_state(n, seed=sum(n))
    for a in range(3):
        if per[a]:
            p = np.concatenate([np.delete(p, -1, a), np.take(p, [0], a)], a)
    sim = HBFlow(n, cfg["h"], np.zeros((3, 2, 3)))
    if any(per):
        sim.set_periodic(per)
    g = Grid(n, cfg["h"], periodic=per, wall_u=np.zeros((3, 2, 3)))
    us_d = torch.tensor(to_device_layout(us), device="cuda")
    p_d = torch.tensor(to_device_layout(p), device="cuda")
    st = sim.project(cfg["dt"], us_d, p_d)
    assert st["converged"], st
    phi = nodes_unique(from_device_layout(p_d.cpu().numpy(), tuple(v + 1 for v in n), 1)[0], g)
    Gp = cell_grad_nodal(nodes_unique(p, g), g)
    w = node_weights(g)
    rhs = nodal_div([us[c] / cfg["dt"] + Gp[c] for c in range(3)], g, w)
    r = rhs - nodal_lap(phi, g)
    r = r - np.sum(w * r) / np.sum(w)
    assert np.max(np.abs(r)) <= 1.1e-10 * np.max(np.abs(rhs))
    sim.close()
