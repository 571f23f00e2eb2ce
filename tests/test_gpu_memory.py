"""Device memory of the mixed contexts: above 2^19 cells the finest level's FP32
Gauss-Seidel reciprocals exist in a batch's cavities, which read them, and not
in a single context, which does not; and the batch's step on such a cavity."""

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


def test_single_contexts_do_without_the_finest_reciprocals():
    from paper_1803_00417_gb300.hbflow import MIXED, Batch, HBFlow

    def held(make):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        x = make()
        torch.cuda.synchronize()
        after = torch.cuda.mem_get_info()[0]
        x.close()
        return before - after

    n, h = (128, 128, 128), 1.0 / 128
    single, batch = (lambda: HBFlow(n, h, precision=MIXED)), (lambda: Batch([n], [h], precision=MIXED))
    held(single), held(batch)  # first use of the device
    extra = held(batch) - held(single)
    assert extra >= 3 * 128 ** 3 * 4 - (2 << 20)  # one FP32 vector, less the allocator's 2 MB


# tolerance: each route's solves stop at 1e-10 of the right-hand side (as the batch's routes, 1e-8 of the largest value)
def test_batch_step_above_the_limit():
    from paper_1803_00417_gb300.hbflow import MIXED, Batch, HBFlow

    cfg = cavity((1024, 640), Re=100.0, Bi=10.0, Pa=1e4, nexp=1.2)
    u, p = random_state(cfg["n"], seed=9)
    B = Batch([cfg["n"]], [cfg["h"]], [cfg["wall_u"]], precision=MIXED)
    sim = HBFlow(cfg["n"], cfg["h"], cfg["wall_u"], precision=MIXED)
    for v in (B.cavity(0), sim):
        v.set_rheology(cfg["K"], cfg["nexp"], cfg["tau_y"], cfg["m"])
        v.set_velocity(u)
        v.set_pressure(p)
    B.set_dt([cfg["dt"]])
    stats = B.step()[0], sim.step(cfg["dt"])
    assert all(s[k]["converged"] for s in stats for k in ("mac", "visc", "nodal")), stats
    for f in ("U", "P"):
        a, b = B.cavity(0).get_field(f), sim.get_field(f)
        assert np.max(np.abs(a - b)) <= 1e-8 * np.max(np.abs(b))
    B.close()
    sim.close()
