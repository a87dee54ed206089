"""The four-column march and the adjoint tiles in the bounds-checked build (a bad
index sets a status bit; the loads and the adjoint's accesses are redirected,
nothing traps), at the edges of strips, groups, rows, bands and tiles.  The
checked library is loaded in child processes."""
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEAD = """
import sys
import torch
from paper_1810_07642_gb300 import _lib, inputs
from paper_1810_07642_gb300.adjoint import _Tape
from paper_1810_07642_gb300.film import FilmBatch, ThinFilm
def film(nx, ny, dtype, field=True, **over):
    h0, th, p = inputs.small_random(nx, ny, seed=nx + ny, amp=0.05)
    return ThinFilm(dict(p, theta_uniform=0.3, **over), h0, th if field else None, dtype=dtype)
bad, runs = [], 0
def done(sim, *what):
    global runs
    runs += 1
    if sim.check():
        bad.append(what + (sim.check(),))
    sim.close()
"""
TAIL = """
print(runs, "runs", bad[:20])
sys.exit(1 if bad else 0)
"""
MARCH = """
for field in (True, False):
    # one strip and several, groups that end a row and that wrap, bands of one row up
    for nx, ny in [(8, 9), (9, 7), (10, 9), (11, 8), (12, 5), (32, 3), (33, 8), (118, 17), (119, 16), (120, 33), (121, 12), (122, 33),
                   (124, 40), (125, 9), (126, 1), (128, 2), (238, 8), (240, 8), (241, 24), (242, 100), (364, 21), (365, 20)]:
        sim = film(nx, ny, "f32", field)
        _lib.use_wide(sim.handle)
        for n in (1, 2, 3, 11):
            sim.step(n)
        done(sim, nx, ny, "f32", field)
    for dtype in ("f32", "f16", "bf16"):
        films = [film(nx, ny, dtype, field) for nx, ny in [(4, 6), (8, 9), (12, 1), (116, 17), (120, 33), (124, 40), (240, 8), (244, 100)]]
        with FilmBatch(films) as batch:
            _lib.use_wide(batch=batch.batch)
            for n in (1, 2, 3, 11):
                batch.step(n)
        for f in films:
            done(f, "batch", f.nx, f.ny, dtype, field)
"""
ADJOINT = """
for nx, ny in [(1, 1), (2, 3), (5, 4), (15, 7), (16, 8), (17, 9), (33, 17), (64, 31)]:
    for dtype in ("f32", "f64", "bf16"):
        for bx in (64, 128, 256):
            for tau in (1.0, 0.8):
                sim = film(nx, ny, dtype, tau=tau)
                _lib.use_tiles(sim.handle, bx)
                tape = _Tape(sim, 5, 2)
                tape.forward()
                tape.backward(torch.ones((ny, nx), device="cuda"), True, True)
                _lib.tf_lbm_tape_destroy(tape.tape)
                tape.tape = None
                done(sim, nx, ny, dtype, bx, tau)
"""


@pytest.mark.parametrize("code", [MARCH, ADJOINT], ids=["march", "adjoint"])
def test_indices_stay_in_bounds(code):
    from paper_1810_07642_gb300 import build
    lib = build.build(checked=True)
    r = subprocess.run([sys.executable, "-c", HEAD + code + TAIL], cwd=ROOT,
                       env=dict(os.environ, TFLBM_LIBRARY=lib, PYTHONPATH=ROOT), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
