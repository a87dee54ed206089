"""Calls on several streams: what a handle keeps from one call to the next may
not depend on the stream that the first one came on."""
import pytest

torch = pytest.importorskip("torch")

from paper_1810_07642_gb300 import _lib, inputs
from paper_1810_07642_gb300.film import ThinFilm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_diagnostics_on_a_second_stream_while_the_first_is_busy(dtype):
    """The first call waits behind other work on its stream; the second comes on
    another one and is done before the first has begun."""
    h0, th, p = inputs.small_random(130, 70, seed=3, amp=0.05)
    other = ThinFilm(p, h0, th, dtype=dtype)
    want = other.diagnostics(1.0, (2, 1))
    sim = ThinFilm(p, h0, th, dtype=dtype)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    out = [torch.zeros(12, dtype=torch.float64, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    with torch.cuda.stream(a):
        torch.cuda._sleep(200_000_000)  # about 0.1 s
    _lib.tf_lbm_diagnostics(sim.handle, 1.0, 2, 1, out[0].data_ptr(), a.cuda_stream)
    _lib.tf_lbm_diagnostics(sim.handle, 1.0, 2, 1, out[1].data_ptr(), b.cuda_stream)
    b.synchronize()
    assert torch.equal(out[1], want)
    a.synchronize()
    assert torch.equal(out[0], want)
