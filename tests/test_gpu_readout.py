"""Read-out kernels at the edges of their tiles: pressure and force (64 x 16
tiles with a halo of 2), diagnostics (units of 32 columns x 16 rows), moments
and the state round trip, on lattices down to one node, against the oracle's
definitions on the exported state.

Tolerances: FP64 1e-11 of the field's largest value (summation order only).
FP32: the pressure sums h - href of |values| <= 0.1 with a stencil weight of
20/3, so its rounding is below 20/3 * 0.1 * 2^-22 = 1.6e-7 against pressures of
gamma * 0.1; 1e-4 relative leaves a factor of 60 over gamma's cancellation.
The diagnostics sum exported FP32 heights exactly (2^-48 a term): 1e-6 covers
h = fl(sum f_l), 2^-22 a node.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1810_07642_gb300 import _lib as L
from paper_1810_07642_gb300 import inputs
from paper_1810_07642_gb300.film import FilmBatch, ThinFilm

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (2, 1), (1, 5), (3, 2), (31, 15), (32, 16), (33, 17), (63, 16), (64, 17), (65, 33), (130, 70)]


def sim_of(nx, ny, dtype, **over):
    h0, th, p = inputs.small_random(nx, ny, seed=nx * 100 + ny, amp=0.05)
    p.update(gx_body=1e-4, gy_body=-2e-4, g=1e-3, **over)
    sim = ThinFilm(p, h0, th, dtype=dtype)
    sim.step(5)
    return sim, O.Config(**{k: v for k, v in p.items() if k in O.Config.__dataclass_fields__}), th


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
def test_pressure_force_and_moments_at_tile_edges(nx, ny, dtype):
    sim, cfg, th = sim_of(nx, ny, dtype)
    f = np.ascontiguousarray(sim.get_state().cpu().numpy())
    p, fx, fy = O.pressure_force(cfg, O.kappa_field(cfg, th), f)
    h, ux, uy = O.moments(cfg, f)
    tol = 1e-11 if dtype == "f64" else 1e-4
    got = dict(sim.pressure_force(), **sim.moments())
    for name, want in dict(p=p, fx=fx, fy=fy, h=h, ux=ux, uy=uy).items():
        scale = np.abs(want).max() + (1e-3 if name in ("fx", "fy", "ux", "uy") else 0)
        assert np.abs(got[name].double().cpu().numpy() - want).max() <= tol * scale, name
    # the state goes out and in unchanged
    g = sim.get_state()
    sim.set_state(g)
    assert torch.equal(sim.get_state(), g)


@pytest.mark.parametrize("dtype", ["f64", "f32", "f16"])
@pytest.mark.parametrize("mode", [(1, 0), (-3, 2), (7, -40)])
def test_diagnostics_of_ragged_batches(dtype, mode):
    sims = [sim_of(nx, ny, dtype)[0] for nx, ny in SIZES]
    batch = FilmBatch(sims)
    rows = batch.diagnostics(1.0, mode).cpu().numpy()
    for (nx, ny), sim, row in zip(SIZES, sims, rows):
        want = reference(sim, nx, ny, mode, dtype)
        tol = 1e-11 if dtype == "f64" else 1e-6
        scale = np.maximum(np.abs(want), nx * ny * (1e-3 if dtype != "f64" else 1.0))
        alone = sim.diagnostics(1.0, mode).cpu().numpy()
        assert np.all(np.abs(row - want) <= tol * scale), (nx, ny, row - want)
        assert np.all(np.abs(alone - want) <= tol * scale), (nx, ny, alone - want)
    batch.close()


def reference(sim, nx, ny, mode, dtype):
    """tf_lbm_diag by its definition from the heights and momenta of the state, in FP64."""
    m = sim.moments()
    h = m["h"].double().cpu().numpy()
    f = sim.get_state().cpu().numpy()
    jx = f[1] + f[2] + f[8] - f[4] - f[5] - f[6]
    jy = f[2] + f[3] + f[4] - f[6] - f[7] - f[8]
    wet = h > 1.0
    x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
    ax, ay = 2 * math.pi * x / nx, 2 * math.pi * y / ny
    ph = 2 * math.pi * (((mode[0] * x) % nx) / nx + ((mode[1] * y) % ny) / ny)
    hw = h * wet
    d = dict(mass=h.sum(), wet_mass=hw.sum(), wet_jx=(wet * jx).sum(), wet_jy=(wet * jy).sum(), wet_area=wet.sum(),
             h_max=h.max(), wet_cos_x=(hw * np.cos(ax)).sum(), wet_sin_x=(hw * np.sin(ax)).sum(),
             wet_cos_y=(hw * np.cos(ay)).sum(), wet_sin_y=(hw * np.sin(ay)).sum(),
             mode_cos=(h * np.cos(ph)).sum(), mode_sin=(h * np.sin(ph)).sum())
    return np.array([float(d[k]) for k in L.DIAG_FIELDS])
