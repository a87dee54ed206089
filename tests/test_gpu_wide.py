"""The four-column march (default at tau = 1 on lattices larger than L2, and of
batches): every strip and band edge, both FP32 layouts between steps, every way
to split a run into calls.

The march runs the node arithmetic of the two-column kernel in the same order
with paired FP32 instructions, which leave the compiler no contraction, so the
states agree bit for bit (tolerance 0).  A batch runs it at any size, which is
how the small lattices here reach it.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1810_07642_gb300 import _lib, inputs
from paper_1810_07642_gb300.film import FilmBatch, ThinFilm

pytestmark = pytest.mark.gpu

# around one and two strips of 120 columns, narrower than the stencil's halo,
# multiples of 4 and not
QUAD = [(8, 9), (12, 5), (116, 17), (120, 33), (124, 40), (240, 8), (244, 100), (364, 21)]
EVEN = [(10, 9), (118, 17), (122, 33), (126, 40), (238, 8), (242, 100), (362, 21)]


def films_of(sizes, dtype, uniform):
    films, specs = [], []
    for i, (nx, ny) in enumerate(sizes):
        h0, th, p = inputs.small_random(nx, ny, seed=nx * 7 + ny, amp=0.05)
        p.update(g=2e-4 * (i % 3), gx_body=1e-5, gy_body=-2e-5, delta=0.7, theta_uniform=math.radians(25.0))
        if i % 4 == 3:
            p.update(n_exp=9, m_exp=3)
        th = None if uniform else th
        specs.append((p, h0, th))
        films.append(ThinFilm(p, h0, th, dtype=dtype))
    return films, specs


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("uniform", [False, True])
@pytest.mark.parametrize("sizes", [QUAD, EVEN], ids=["quad", "even"])
def test_batches_of_small_domains_give_the_two_column_bits(dtype, uniform, sizes):
    films, specs = films_of(sizes, dtype, uniform)
    batch = FilmBatch(films)
    for n in (1, 2, 3, 17):
        batch.step(n)
    for (p, h0, th), f in zip(specs, films):
        ref = ThinFilm(p, h0, th, dtype=dtype)
        ref.set_launch(pipeline=3, block_x=64, rows=7)
        ref.step(23)
        assert f.time == 23 and f.check() == 0
        assert torch.equal(f.get_state(), ref.get_state()), (p["nx"], p["ny"])
        ref.close()
    batch.close()


@pytest.mark.parametrize("dtype,nx,ny", [("f32", 1204, 950), ("f32", 1206, 950), ("f32", 1203, 951),
                                         ("f16", 1204, 950), ("bf16", 1204, 950)])
def test_large_lattice_splits_and_bits(dtype, nx, ny):
    h0, th, p = inputs.small_random(nx, ny, seed=3, amp=0.05)
    p.update(g=2e-4, gx_body=1e-5, gy_body=-2e-5)
    states = []
    for split in ((12,), (1, 1, 2, 8), (3, 9), None):
        sim = ThinFilm(p, h0, th, dtype=dtype)
        m0 = sim.mass()
        if split is None:
            _lib.use_tiles(sim.handle, 256)  # tiles run the same node arithmetic
            sim.step(12)
        else:
            for n in split:
                sim.step(n)
                assert sim.check() == 0  # the state between calls is populations
        assert abs(sim.mass() - m0) <= 1e-6 * m0
        states.append(sim.get_state())
        sim.close()
    for s in states[1:]:
        assert torch.equal(states[0], s)


def test_against_the_oracle():
    """Parity tolerance of FP32 (1e-5 of h after 60 steps)."""
    films, specs = films_of([(244, 100), (242, 50)], "f32", False)
    batch = FilmBatch(films)
    batch.step(60)
    for (p, h0, th), f in zip(specs, films):
        cfg = O.Config(**{k: v for k, v in p.items() if k in O.Config.__dataclass_fields__})
        ho = O.run(cfg, h0, th, 60)[1]
        h = f.h().double().cpu().numpy()
        assert np.abs(h - ho).max() <= 1e-5 * np.abs(ho).max()
    batch.close()


def test_graph_chunks_and_single_steps_in_between():
    films, specs = films_of(QUAD, "f32", False)
    batch = FilmBatch(films)
    assert batch.launch["graph_chunk"] == 64  # few nodes: steps replay a graph of 64
    batch.step(65)
    films[2].step(1)
    batch.step(66)
    for i, ((p, h0, th), f) in enumerate(zip(specs, films)):
        ref = ThinFilm(p, h0, th)
        ref.set_launch(pipeline=3, block_x=128, rows=9)
        ref.step(131 + (i == 2))
        assert torch.equal(f.get_state(), ref.get_state()), i
        ref.close()
    batch.close()
