"""What a gradient tape may hold: nothing where no gradient can be asked for,
and no more than 4 GiB of records where recomputing them takes less."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1810_07642_gb300 import _lib, inputs
from paper_1810_07642_gb300.adjoint import evolve
from paper_1810_07642_gb300.film import ThinFilm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_a_run_without_gradients_makes_no_tape(monkeypatch, tau):
    h0, th, p = inputs.small_random(130, 70, seed=1, amp=0.05)
    p.update(tau=tau)
    theta, hh = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in (th, h0))
    with_tape = evolve(theta.clone().requires_grad_(), hh, p, 20).detach()

    def no_tape(*_):
        raise AssertionError("a tape was made")

    monkeypatch.setattr(_lib, "tf_lbm_tape_create", no_tape)
    want = ThinFilm(p, hh, theta)
    want.step(20)
    assert torch.equal(evolve(theta, hh, p, 20), want.h())
    with torch.no_grad():
        got = evolve(theta.clone().requires_grad_(), hh.clone().requires_grad_(), p, 20)
    assert torch.equal(got, want.h()) and torch.equal(got, with_tape)
    with pytest.raises(AssertionError):
        evolve(theta, hh.clone().requires_grad_(), p, 20)


def test_refusals_are_kept_without_gradients():
    h0, th, p = inputs.small_random(16, 16, seed=1)
    theta, hh = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in (th, h0))
    with pytest.raises(_lib.TfLbmError):
        evolve(theta, hh, p, 0)
    with pytest.raises(_lib.TfLbmError):
        evolve(theta, hh, dict(p, forcing=1), 3)


def test_records_kept_stay_below_four_gigabytes():
    """512^2, 2000 steps: 6.3 GB of records, 0.6 GB in segments; and the
    gradient is that of explicit segments."""
    h0, th, p = inputs.small_random(512, 512, seed=2, amp=0.02)
    grads = []
    for every in (0, 100):
        theta = torch.tensor(th, dtype=torch.float32, device="cuda", requires_grad=True)
        hh = torch.tensor(h0, dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        h = evolve(theta, hh, p, 2000, every=every)
        assert before - torch.cuda.mem_get_info()[0] <= 4 << 30
        grads.append(torch.autograd.grad((h * h).sum(), theta)[0])
    # records kept and recomputed are the same bits
    assert torch.equal(grads[0], grads[1]) and np.isfinite(grads[0].cpu().numpy()).all()
