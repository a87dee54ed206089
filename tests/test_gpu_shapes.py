"""Launch shapes: what a run gives may not depend on how it is split into calls
or on which march the four-column march was put in place of, and a shape that
the library chose is kept by reading it and setting it again.

The four-column, two-column and tile kernels run the same node arithmetic with
paired FP32 instructions, which leave the compiler no contraction: states agree
bit for bit (tolerance 0).
"""
import pytest

torch = pytest.importorskip("torch")

from paper_1810_07642_gb300 import _lib, inputs
from paper_1810_07642_gb300.film import FilmBatch, ThinFilm

pytestmark = pytest.mark.gpu


def film(nx, ny, dtype="f32", tau=1.0, field=True):
    h0, th, p = inputs.small_random(nx, ny, seed=nx + 3 * ny, amp=0.05)
    p.update(tau=tau, g=2e-4, gx_body=1e-5, gy_body=-2e-5, theta_uniform=0.3)
    return ThinFilm(p, h0, th if field else None, dtype=dtype)


# ragged and whole groups of four columns; the one-column march beneath
@pytest.mark.parametrize("nx,ny", [(244, 100), (242, 51), (121, 60)])
@pytest.mark.parametrize("base", [dict(pipeline=1, block_x=64, rows=16), dict(pipeline=2, block_x=128, rows=30)])
def test_one_step_runs_of_the_four_column_march_keep_its_bits(nx, ny, base):
    states = []
    for split in ((9,), (1,) * 9, (1, 2, 1, 5)):
        sim = film(nx, ny)
        sim.set_launch(graph_chunk=0, **base)
        _lib.use_wide(sim.handle)
        for n in split:
            sim.step(n)
        states.append(sim.get_state())
        sim.close()
    assert torch.equal(states[0], states[1]) and torch.equal(states[0], states[2])


@pytest.mark.parametrize("sizes", [[(244, 100), (120, 33)], [(240, 51), (116, 17), (12, 9)]])
def test_one_step_runs_of_a_batch_keep_its_bits(sizes):
    states = []
    for split in ((9,), (1,) * 9, (1, 2, 1, 5)):
        films = [film(nx, ny) for nx, ny in sizes]
        with FilmBatch(films) as batch:
            batch.set_launch(pipeline=1, block_x=64, rows=16, graph_chunk=0)
            _lib.use_wide(batch=batch.batch)
            for n in split:
                batch.step(n)
            states.append([f.get_state() for f in films])
        [f.close() for f in films]
    for s in states[1:]:
        assert all(torch.equal(a, b) for a, b in zip(states[0], s))


@pytest.mark.parametrize("dtype,tau", [("f32", 0.8), ("f64", 1.0), ("bf16", 1.3)])
def test_setting_what_was_read_keeps_the_kernel(dtype, tau):
    """Off tau = 1, and in FP64, tiles and the march that the fields describe
    differ in the last bits, which shows the kernel; default and tuned shape,
    set as they are, with another graph_chunk, and after other shapes."""
    sim = film(300, 200, dtype, tau)
    s0 = sim.get_state()

    def after(steps=40):
        sim.set_state(s0)
        sim.step(steps)
        return sim.get_state()

    for tuned in (False, True):
        shape, want = sim.launch, after()
        sim.set_launch(**shape)
        assert torch.equal(after(), want)
        sim.set_launch(graph_chunk=8)
        assert torch.equal(after(), want) and sim.launch == dict(shape, graph_chunk=8)
        sim.set_launch(block_x=128, rows=23, pipeline=1)
        assert tuned or not torch.equal(after(), want)
        sim.set_launch(**shape)
        assert torch.equal(after(), want)
        sim.set_state(s0)
        assert sim.tune(4) == sim.launch
    sim.close()


def test_setting_what_was_read_keeps_the_kernel_of_a_batch():
    """The number of work items shows the kernel."""
    films = [film(nx, ny) for nx, ny in [(512, 256)] * 6 + [(1024, 512)]]
    with FilmBatch(films) as batch:
        for _ in range(2):
            shape, items = batch.launch, batch.items
            batch.set_launch(**shape)
            assert batch.items == items
            batch.set_launch(graph_chunk=4, queue=0)
            if not shape["queue"]:
                assert batch.items == items
            batch.set_launch(block_x=64, rows=1, pipeline=1)
            assert batch.items > items
            batch.set_launch(**shape)
            assert batch.items == items and batch.launch == shape
            batch.step(3)
            assert batch.tune(4) == batch.launch
    [f.close() for f in films]


# widths that are multiples of 4 beside one that is not, down to lattices whose
# moment rows would not fit a population buffer: no four-column march
@pytest.mark.parametrize("sizes", [[(240, 64), (242, 100), (64, 33), (122, 9)], [(32, 3), (242, 20), (8, 40)],
                                   [(32, 2), (242, 20)], [(32, 1), (122, 7)], [(4, 9), (242, 20)]])
def test_batches_that_mix_layouts(sizes):
    films = [film(nx, ny) for nx, ny in sizes]
    with FilmBatch(films) as batch:
        with pytest.raises(ValueError):
            _lib.use_wide(batch=batch.batch)
        for n in (1, 2, 3, 17):
            batch.step(n)
    for f, (nx, ny) in zip(films, sizes):
        ref = film(nx, ny)
        ref.set_launch(pipeline=3, block_x=64, rows=7)
        ref.step(23)
        assert f.check() == 0 and torch.equal(f.get_state(), ref.get_state()), (nx, ny)
        ref.close()
        f.close()


# 16-bit domains whose strips are mostly empty: two columns where there are many,
# four where there are few; items = strips x bands of the march in use
@pytest.mark.parametrize("nx,ny,count,four", [(8, 3000, 12, False), (8, 700, 3, True), (64, 3000, 12, True)])
def test_narrow_16_bit_batches(nx, ny, count, four):
    films = [film(nx, ny, "f16", field=False) for _ in range(count)]
    with FilmBatch(films) as batch:
        default = batch.items
        batch.set_launch(queue=1)
        two = batch.items
        assert (default != two) == four
        batch.step(2)
        assert all(f.check() == 0 for f in films)
    [f.close() for f in films]


# ragged lattices on either side of the rules: tiles, the four-column march with
# runs of at least eight steps, the two-column march (two strips); odd: no two
# columns.  FP32 at tau = 1: the same bits whatever the kernel.
@pytest.mark.parametrize("nx,ny", [(1030, 1040), (1030, 1262), (126, 13000), (242, 9090), (1205, 1330), (362, 4000)])
def test_ragged_runs_of_any_length_give_the_same_bits(nx, ny):
    states = []
    for split in ((17,), (3, 8, 1, 5), (7, 10), (2,) * 8 + (1,), None):
        sim = film(nx, ny)
        if split is None:
            _lib.use_tiles(sim.handle, 256, graph_chunk=4)
            split = (17,)
        for n in split:
            sim.step(n)
        assert sim.check() == 0 and sim.time == 17
        states.append(sim.get_state())
        sim.close()
    assert all(torch.equal(states[0], s) for s in states[1:])
