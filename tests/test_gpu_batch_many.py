"""Batches of more cavities than clusters of two blocks fit the GPU (77 and
more): each cavity's V-cycle tail is one block, and levels that its shared
memory cannot hold run level by level.  Against the same batch level by level,
and one cavity against the oracle.

Tolerances: 1e-8 of the largest value between the routes and 1e-6 relative L2
against the oracle, as the batch's other tests in mixed precision."""

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


@pytest.mark.parametrize("precision", [0, 1])
def test_many_cavities(precision):
    from paper_1803_00417_gb300.hbflow import Batch

    sizes = [((64, 64), (48, 32), (64, 32), (16, 16))[i % 4] for i in range(80)]
    cfgs = [cavity(n, Re=100.0, Bi=1.0 + i % 7, Pa=1e4, nexp=1.2) for i, n in enumerate(sizes)]
    states = [random_state(n, seed=i) for i, n in enumerate(sizes)]
    outs = []
    for tail in (None, 0):
        B = Batch([c["n"] for c in cfgs], [c["h"] for c in cfgs], [c["wall_u"] for c in cfgs], precision=precision)
        if tail is not None:
            B.set_tail(tail)
        for i, c in enumerate(cfgs):
            v = B.cavity(i)
            v.set_rheology(c["K"], c["nexp"], c["tau_y"], c["m"])
            v.set_velocity(states[i][0])
            v.set_pressure(states[i][1])
        B.set_dt([c["dt"] for c in cfgs])
        st = B.step()
        assert all(s[k]["converged"] for s in st for k in ("mac", "visc", "nodal")), st
        outs.append([np.concatenate([B.cavity(i).get_field("U"), B.cavity(i).get_field("P")]) for i in range(80)])
        if tail is None:
            c = cfgs[4]
            ref = step(Grid(c["n"], c["h"], wall_u=c["wall_u"]), *states[4], c["dt"],
                       Rheology(c["K"], c["nexp"], c["tau_y"], c["m"]))
            got, want = np.array(B.cavity(4).velocity()), np.array(ref.u)
            assert np.linalg.norm(got - want) <= 1e-6 * np.linalg.norm(want)
        B.close()
    for a, b in zip(*outs):
        assert np.max(np.abs(b - a)) <= 1e-8 * np.max(np.abs(a))
