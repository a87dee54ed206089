"""Gradients at the edges of every tile shape, which a tape picks by the lattice's
size: here each lattice runs each of them, forward and adjoint.

Tolerances: those of the tape tests: FP64 1e-9 of the largest entry against the
oracle's gradient (summation order only), FP32 1e-3.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1810_07642_gb300 import _lib, inputs
from paper_1810_07642_gb300.adjoint import _Tape
from paper_1810_07642_gb300.film import ThinFilm

pytestmark = pytest.mark.gpu

# one node, narrower than the four nested stencils, one less / equal / one more
# than the 16 x 8, 16 x 16 and 32 x 16 tiles
SIZES = [(1, 1), (2, 3), (5, 4), (15, 7), (16, 8), (17, 9), (31, 15), (32, 16), (33, 17), (64, 31)]


def oracle_gradient(p, h0, th, steps, target):
    cfg = O.Config(**{k: v for k, v in p.items() if k in O.Config.__dataclass_fields__})

    def seed(f):
        h = f.sum(0)
        return 0.5 * float(((h - target) ** 2).sum()), np.broadcast_to(h - target, f.shape).copy()

    _, gth, gh0, _ = O.loss_gradient(cfg, h0, th, steps, seed)
    return gth, gh0


@pytest.mark.parametrize("block_x", [64, 128, 256])
@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_gradient_in_every_tile_shape(nx, ny, tau, block_x):
    h0, th, p = inputs.small_random(nx, ny, seed=7 * nx + ny, amp=0.1)
    p.update(tau=tau, g=1e-3, delta=0.8, gx_body=1e-4)
    steps, target = 12, np.random.default_rng(2).uniform(0.9, 1.1, h0.shape)
    want = oracle_gradient(p, h0, th, steps, target)
    for dtype, every, tol in (("f64", 0, 1e-9), ("f64", 5, 1e-9), ("f32", 0, 1e-3), ("f32", 5, 1e-3)):
        sim = ThinFilm(p, h0, th, dtype=dtype)
        _lib.use_tiles(sim.handle, block_x)
        tape = _Tape(sim, steps, every)
        tape.forward()
        got = tape.backward(sim.h() - torch.tensor(target, dtype=sim.tdtype, device="cuda"), True, True)
        for name, a, b in zip(("theta", "h0"), got, want):
            if dtype == "f32" and name == "theta" and nx * ny == 1:
                continue  # a 1 x 1 film has no pressure gradient
            assert np.abs(a.double().cpu().numpy() - b).max() <= tol * max(np.abs(b).max(), 1e-12), (name, dtype, every)
        tape.close()
