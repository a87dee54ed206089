"""The tile adjoint at the edges of its tiles and of the tape's segments.

Tolerances: those of the tape tests: FP64 1e-9 of the largest entry against the
oracle's gradient (summation order only), FP32 1e-3.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1810_07642_gb300 import inputs
from paper_1810_07642_gb300.adjoint import evolve

pytestmark = pytest.mark.gpu

# one node, narrower than the four nested stencils, around the 16 x 8, 16 x 16
# and 32 x 16 tiles; the last has more tiles than SMs in every shape
SIZES = [(1, 1), (2, 3), (5, 4), (15, 7), (16, 8), (17, 9), (33, 17), (64, 31)]


def oracle_grads(p, h0, th, T, tgt):
    cfg = O.Config(**{k: v for k, v in p.items() if k in O.Config.__dataclass_fields__})

    def seed(f):
        h = f.sum(0)
        return 0.5 * float(((h - tgt) ** 2).sum()), np.broadcast_to(h - tgt, f.shape).copy()

    return O.loss_gradient(cfg, h0, th, T, seed)


def gradients(p, h0, th, T, tgt, dtype, every):
    td = torch.float64 if dtype == "f64" else torch.float32
    theta = torch.tensor(th, dtype=td, device="cuda", requires_grad=True)
    hh = torch.tensor(h0, dtype=td, device="cuda", requires_grad=True)
    h = evolve(theta, hh, p, T, dtype=dtype, every=every)
    loss = 0.5 * ((h - torch.tensor(tgt, dtype=td, device="cuda")) ** 2).sum()
    return [g.double().cpu().numpy() for g in torch.autograd.grad(loss, (theta, hh))]


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_gradient_at_tile_edges(nx, ny, tau):
    h0, th, p = inputs.small_random(nx, ny, seed=7 * nx + ny, amp=0.1)
    p.update(tau=tau, g=1e-3, delta=0.8, gx_body=1e-4)
    T = 12
    tgt = np.random.default_rng(2).uniform(0.9, 1.1, h0.shape)
    _, gth_o, gh0_o, _ = oracle_grads(p, h0, th, T, tgt)
    scale_th = max(np.abs(gth_o).max(), 1e-12)  # a 1 x 1 film has no pressure gradient
    for every in (0, 1, 5, 12):  # all records kept; segments of one, with a remainder, whole
        gth, gh0 = gradients(p, h0, th, T, tgt, "f64", every)
        assert np.abs(gth - gth_o).max() <= 1e-9 * scale_th, every
        assert np.abs(gh0 - gh0_o).max() <= 1e-9 * np.abs(gh0_o).max(), every
    gth, gh0 = gradients(p, h0, th, T, tgt, "f32", 0)
    if nx * ny > 1:
        assert np.abs(gth - gth_o).max() <= 1e-3 * scale_th
    assert np.abs(gh0 - gh0_o).max() <= 1e-3 * np.abs(gh0_o).max()


@pytest.mark.parametrize("tau", [1.0, 0.9])
def test_fp32_gradient_on_more_tiles_than_stay_resident(tau):
    """520 x 500: above three 32 x 16 tiles an SM the FP32 kernel is another
    instantiation."""
    h0, th, p = inputs.small_random(520, 500, seed=3, amp=0.05)
    p.update(tau=tau)
    tgt = np.random.default_rng(4).uniform(0.9, 1.1, h0.shape)
    want = gradients(p, h0, th, 10, tgt, "f64", 0)
    for every in (0, 4):
        got = gradients(p, h0, th, 10, tgt, "f32", every)
        for a, b in zip(got, want):
            assert np.abs(a - b).max() <= 1e-3 * np.abs(b).max()
