"""Default shapes of lattices near the rules that choose the kernel, against the
oracle: long lattices of a few rows or columns, which tiles overhang (some run
tiles, some a march), and the sizes around the smallest FP64 tiles.

Tolerances: those of the parity tests (relative L-infinity on h, 20 steps): FP32
1e-5, FP64 1e-11, 16-bit storage 1e-3; relative mass drift 1e-6.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1810_07642_gb300 import inputs
from paper_1810_07642_gb300.film import ThinFilm

pytestmark = pytest.mark.gpu

TOL = {"f32": 1e-5, "f64": 1e-11, "f16": 1e-3}


def compare(nx, ny, dtype, tau, steps=20):
    h0, th, p = inputs.small_random(nx, ny, seed=nx + ny, amp=0.05)
    p.update(tau=tau, g=2e-4, gx_body=2e-5, gy_body=-1e-5)
    cfg = O.Config(**{k: v for k, v in p.items() if k in O.Config.__dataclass_fields__})
    ho = O.run(cfg, h0, th, steps)[1]
    sim = ThinFilm(p, h0, th, dtype=dtype)
    m0 = sim.mass()
    sim.step(steps)
    assert sim.check() == 0
    assert np.abs(sim.h().double().cpu().numpy() - ho).max() <= TOL[dtype] * np.abs(ho).max()
    assert abs(sim.mass() - m0) <= 1e-6 * m0
    sim.close()


@pytest.mark.parametrize("nx,ny", [(100000, 3), (65000, 17), (40000, 9), (20000, 9), (30000, 3), (60000, 20), (20000, 24),
                                   (30000, 33), (3, 60000), (7, 20000)])
@pytest.mark.parametrize("dtype,tau", [("f32", 1.0), ("f32", 0.8), ("f64", 0.8), ("f16", 0.8)])
def test_long_lattices(nx, ny, dtype, tau):
    compare(nx, ny, dtype, tau)


@pytest.mark.parametrize("nx,ny", [(250, 190), (304, 383), (305, 385), (512, 512), (1030, 1040)])
@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_fp64_tile_shapes(nx, ny, tau):
    compare(nx, ny, "f64", tau)


# 64 x 4 tiles on few of them, 64 x 16 from half the SMs on
@pytest.mark.parametrize("nx,ny", [(64, 4), (65, 5), (63, 37), (321, 190), (321, 260), (257, 511)])
def test_fp64_pressure_and_force_in_either_tile(nx, ny):
    h0, th, p = inputs.small_random(nx, ny, seed=3, amp=0.05)
    p.update(gx_body=1e-4, gy_body=-2e-4, g=1e-3)
    sim = ThinFilm(p, h0, th, dtype="f64")
    sim.step(3)
    cfg = O.Config(**{k: v for k, v in p.items() if k in O.Config.__dataclass_fields__})
    f = np.ascontiguousarray(sim.get_state().cpu().numpy())
    got = sim.pressure_force()
    for name, want in zip(("p", "fx", "fy"), O.pressure_force(cfg, O.kappa_field(cfg, th), f)):
        assert np.abs(got[name].cpu().numpy() - want).max() <= 1e-11 * np.abs(want).max(), name
