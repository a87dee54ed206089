"""The tile kernel at the edges of its tiles against the oracle.

Tolerances: those of the parity tests (relative L-infinity on h, 60 steps):
FP32 1e-5, FP64 1e-11, 16-bit storage 1e-3; relative mass drift 1e-6.
"""
import math
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1810_07642_gb300 import _lib, inputs
from paper_1810_07642_gb300.film import ThinFilm

pytestmark = pytest.mark.gpu

TOL = {"f32": 1e-5, "f64": 1e-11, "f16": 1e-3, "bf16": 1e-3}
# one node, narrower than the stencil, one less / equal / one more than the
# 16 x 8, 16 x 16 and 32 x 16 tiles
SIZES = [(1, 1), (2, 9), (3, 3), (15, 7), (16, 8), (17, 9), (31, 15), (32, 16), (33, 17), (130, 70)]


def compare(nx, ny, dtype, tau, forcing, theta_field):
    h0, th, p = inputs.small_random(nx, ny, seed=nx * 100 + ny, amp=0.05)
    p.update(tau=tau, g=2e-4, gx_body=2e-5, gy_body=-1e-5, forcing=forcing)
    cfg = O.Config(**{k: v for k, v in p.items() if k in O.Config.__dataclass_fields__})
    ho = O.run(cfg, h0, th if theta_field else math.radians(20.0), 60)[1]
    if not theta_field:
        p["theta_uniform"] = math.radians(20.0)
    for block_x in (64, 128, 256):
        sim = ThinFilm(p, h0, th if theta_field else None, dtype=dtype)
        _lib.use_tiles(sim.handle, block_x, graph_chunk=4)
        m0 = sim.mass()
        sim.step(60)
        h = sim.h().double().cpu().numpy()
        assert sim.check() == 0
        assert np.abs(h - ho).max() <= TOL[dtype] * np.abs(ho).max(), block_x
        assert abs(sim.mass() - m0) <= 1e-6 * m0
        sim.close()


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("dtype", ["f32", "f64", "f16", "bf16"])
def test_tile_edges(nx, ny, dtype):
    for tau, forcing, theta_field in ((1.0, 0, True), (0.8, 0, False), (1.0, 1, False), (1.3, 1, True)):
        compare(nx, ny, dtype, tau, forcing, theta_field)


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
def test_tiles_give_the_two_column_march_bit_for_bit(dtype):
    """Same node arithmetic in the same order (paired FP32 instructions, no
    contraction left to the compiler), so the default shape of a small lattice
    and the march it reports agree exactly at tau = 1.  520 x 510: the
    four-resident form of the 32 x 16 tiles too."""
    for nx, ny in ((130, 70), (520, 510)):
        h0, th, p = inputs.small_random(nx, ny, seed=5, amp=0.05)
        p.update(g=2e-4, gx_body=1e-5)
        states = []
        for shape in (None, 256, 64, dict(pipeline=3, block_x=128, rows=16)):
            sim = ThinFilm(p, h0, th, dtype=dtype)
            if isinstance(shape, int):
                _lib.use_tiles(sim.handle, shape)
            elif shape:
                sim.set_launch(**shape)
            sim.step(50)
            states.append(sim.get_state())
            sim.close()
        for s in states[1:]:
            assert torch.equal(states[0], s)


def test_tile_launch_reporting():
    h0, th, p = inputs.small_random(200, 120, seed=4)
    sim = ThinFilm(p, h0, th)
    assert sim.launch["pipeline"] == 3  # the march that the fields describe
    with pytest.raises(Exception):
        sim.set_launch(pipeline=4, block_x=128)
    sim.step(3)
    sim.set_launch(**dict(sim.launch, pipeline=1))
    assert sim.launch["pipeline"] == 1
    sim.step(3)
    assert sim.time == 6


def test_tile_indices_stay_in_bounds():
    """The bounds-checked build over the same lattices (a bad index sets a
    status bit and is redirected; nothing traps)."""
    from paper_1810_07642_gb300 import build
    lib = build.build(checked=True)
    code = """
import sys
from paper_1810_07642_gb300 import _lib, inputs
from paper_1810_07642_gb300.film import ThinFilm
bad = []
for nx, ny in %r:
    for dtype in ("f32", "f64", "bf16"):
        for bx in (64, 128, 256):
            h0, th, p = inputs.small_random(nx, ny, seed=1, amp=0.05)
            sim = ThinFilm(dict(p, tau=0.9), h0, th, dtype=dtype)
            _lib.use_tiles(sim.handle, bx)
            sim.step(5)
            if sim.check():
                bad.append((nx, ny, dtype, bx, sim.check()))
            sim.close()
print(bad)
sys.exit(1 if bad else 0)
""" % (SIZES,)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, env=dict(os.environ, TFLBM_LIBRARY=lib, PYTHONPATH=root),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
