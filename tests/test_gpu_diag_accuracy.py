"""The sums of the film diagnostics against exact sums of the same FP32 heights
and momenta.

Tolerances, in units of sum |addend|: a plain sum is the exact sum rounded to a
double once per merge of a block's (sum, compensation): 2^-52.  A Fourier sum
takes cos and sin of 2 pi x / n in double: 2 ulp of the function (2 * 2^-53) and
its argument's rounding (pi * 2 * 2^-53), 4.2 * 2^-52, below 6 * 2^-52; the mode's
phase has two such factors, 12 * 2^-52.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1810_07642_gb300 import inputs
from paper_1810_07642_gb300.film import FilmBatch, ThinFilm

pytestmark = pytest.mark.gpu

ULP = 2.0 ** -52
WET = 0.5


def exact_sum(v, w=None):
    """Sum of v (float32), or of v times the long doubles w, without rounding."""
    v = v.astype(np.float64).ravel()
    if w is None:
        return math.fsum(v)
    w = np.broadcast_to(w, (v.size,)) if w.ndim == 1 else w.ravel()
    hi = w.astype(np.float64)
    lo = (w - hi).astype(np.float64)
    top = hi.astype(np.float32).astype(np.float64)  # 24 + 24 bits and 24 + 29 bits: exact products
    return math.fsum(np.concatenate([v * top, v * (hi - top), v * lo]))


def angles(n, k=1):
    a = 8 * np.arctan(np.longdouble(1)) * ((k * np.arange(n)) % n).astype(np.longdouble) / n
    return np.cos(a), np.sin(a)


def check(sim, row, mode):
    nx, ny = sim.nx, sim.ny
    h = sim.moments(("h",))["h"].cpu().numpy()
    f = sim.get_state().cpu().numpy()[1:].astype(np.float32)
    f = np.concatenate([f[:1], f])  # f[l], l = 1 .. 8, as stored
    jx = ((f[1] + f[2]) + f[8]) - ((f[4] + f[5]) + f[6])
    jy = ((f[2] + f[3]) + f[4]) - ((f[6] + f[7]) + f[8])
    wet = h > np.float32(WET)
    hw = np.where(wet, h, np.float32(0))
    (cx, sx), (cy, sy) = angles(nx), angles(ny)
    (ca, sa), (cb, sb) = angles(nx, mode[0]), angles(ny, mode[1])
    at = lambda a, b: np.ascontiguousarray(np.broadcast_to(a[None, :], (ny, nx)) if b is None else
                                           np.broadcast_to(b[:, None], (ny, nx)))
    total, wet_total = exact_sum(np.abs(h)), exact_sum(hw)
    plain = {0: (h, total), 1: (hw, wet_total), 2: (jx * wet, exact_sum(np.abs(jx * wet))),
             3: (jy * wet, exact_sum(np.abs(jy * wet)))}
    for k, (v, scale) in plain.items():
        assert abs(row[k] - exact_sum(v)) <= ULP * scale, (k, row[k], exact_sum(v))
    assert row[4] == wet.sum() and row[5] == h.max()
    for k, w in {6: at(cx, None), 7: at(sx, None), 8: at(None, cy), 9: at(None, sy)}.items():
        assert abs(row[k] - exact_sum(hw, w)) <= 6 * ULP * wet_total, (k, row[k], exact_sum(hw, w))
    cos = ca[None, :] * cb[:, None] - sa[None, :] * sb[:, None]
    sin = sa[None, :] * cb[:, None] + ca[None, :] * sb[:, None]
    for k, w in {10: cos, 11: sin}.items():
        assert abs(row[k] - exact_sum(h, w)) <= 12 * ULP * total, (k, row[k], exact_sum(h, w))


# a batch gives a domain 64 blocks: columns of 16 to 150 rows to a sum
@pytest.mark.parametrize("nx,ny", [(31, 17), (256, 128), (512, 2048), (4096, 256), (8192, 150)])
def test_sums_are_exact_to_the_rounding_of_the_result(nx, ny):
    rng = np.random.default_rng(nx + ny)
    # a thick film over a precursor; the heights repeat every 128 rows and do
    # not depend on x in the first domain, so that errors of a sum do not cancel
    rows = rng.uniform(0.07, 40.0, min(ny, 128)).astype(np.float32)
    h0 = np.repeat(np.resize(rows, ny)[:, None], nx, 1)
    p = inputs._params(nx, ny)
    films = [ThinFilm(p, h0), ThinFilm(p, rng.uniform(0.07, 40.0, (ny, nx)).astype(np.float32))]
    f = films[1].get_state()
    f[1:] += 0.1 * torch.rand(f[1:].shape, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda",
                              dtype=f.dtype)
    films[1].set_state(f)
    mode = (3, -2)
    with FilmBatch(films) as batch:
        got = batch.diagnostics(WET, mode).cpu().numpy()
    for sim, row in zip(films, got):
        check(sim, row, mode)
        check(sim, sim.diagnostics(WET, mode).cpu().numpy(), mode)
        sim.close()


def test_sums_beyond_the_range_of_a_float():
    """A film that has run away: heights that a float holds, their sum not."""
    p = inputs._params(1024, 2048)
    sim = ThinFilm(p, np.full((2048, 1024), 3e37, np.float32))
    with FilmBatch([sim]) as batch:
        for row in (batch.diagnostics(WET)[0], sim.diagnostics(WET)):
            row = row.cpu().numpy()
            want = float(np.float32(3e37)) * 2048 * 1024
            assert abs(row[0] - want) <= ULP * want and row[5] == float(np.float32(3e37))
            assert np.isfinite(row).all()
    sim.close()
