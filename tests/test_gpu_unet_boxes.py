"""The network on boxes whose levels are no multiple of the convolution and
weight-gradient tiles (x extents of 24, 40 and 72: 12 to 3 cells on the coarse
levels; one axis of a single coarse cell), forward and gradients of both
convolution paths against the CPU reference network.

Tolerances: those of the same comparison on the cubic boxes (bf16 operands of
11 convolutions: 2e-2 forward, 6e-2 for the gradients)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle.unet as U  # noqa: E402
from test_gpu_unet import from_gpu_params, rel, spatial_to_flat, to_gpu_params  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_00417_gb300 import build

    build.build()


@pytest.mark.parametrize("n", [(40, 24), (24, 40, 16), (72, 8, 24), (16, 48, 40)])
@pytest.mark.parametrize("path", [0, 1])
def test_boxes_match_reference(n, path):
    from paper_1803_00417_gb300.hbflow import UNet

    d = len(n)
    rng = np.random.default_rng(sum(n))
    params = U.init_params(d, seed=sum(n))
    for p in params:
        p[1] = (p[1] + rng.normal(size=p[1].shape) * 0.05).astype(np.float32).astype(np.float64)
        p[0] = p[0].astype(np.float32).astype(np.float64)
    x, t = rng.normal(size=n), rng.normal(size=n)
    net = UNet(n, train=True)
    net.set_tensor_path(path)
    net.set_params(to_gpu_params(params))
    xd = torch.tensor(spatial_to_flat(x).astype(np.float32), device="cuda")
    td = torch.tensor(spatial_to_flat(t).astype(np.float32), device="cuda")
    yd, gy = torch.empty_like(xd), torch.empty_like(xd)
    net.zero_grads()
    net.forward(xd, yd)
    net.loss(td, torch.ones_like(xd), gy)
    net.backward(gy)
    net.tensor_status()
    g_gpu = from_gpu_params(net.get_grads(), d)
    net.close()
    y_ref, tape = U.forward(params, U.bf16(x)[..., None], keep=True)
    assert rel(yd.cpu().numpy(), spatial_to_flat(y_ref[..., 0])) < 2e-2
    _, gy_ref = U.mse_loss(y_ref, t[..., None], np.ones(n + (1,)))
    g_ref = U.backward(params, tape, gy_ref)
    for k in range(len(params)):
        for w in (0, 1):
            assert rel(g_gpu[k][w], g_ref[k][w]) < 6e-2, (k, w)
