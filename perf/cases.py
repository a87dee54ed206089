"""Timed cases: the work that a user of this library has it do, through ThinFilm, FilmBatch and evolve.

A case is a dict; its "kind" says what one pass is:
  film       step(steps), then the film height: a simulation advanced between two read-outs
  sweep      FilmBatch.step(steps) over many uneven domains, then every domain's height
  gradient   evolve() and its backward pass: heights, dL/dtheta and dL/dh0
  readout    moments() and pressure_force() of a state: what a run writes for plots
  restart    set_state() of a saved state, then get_state(): checkpoint and resume
  diagnose   FilmBatch.diagnostics(): the monitoring numbers of a parameter sweep

Heights and contact angles are drawn on the GPU from the seed alone, shaped like the workloads of inputs.py:
"ripple" (one sinusoidal mode on a flat film), "drop" (a spherical cap on a precursor film) and "noise" (a noisy film
on a striped and patched substrate).
"""
import math

import torch

from paper_1810_07642_gb300.adjoint import evolve
from paper_1810_07642_gb300.film import FilmBatch, ThinFilm

HSTAR = 0.07
BASE = dict(gamma=0.01, g=0.0, delta=1.0, hstar=HSTAR, n_exp=3, m_exp=2, pi_sign=1, gx_body=0.0, gy_body=0.0)
CX = (0, 1, 1, 0, -1, -1, -1, 0, 1)
CY = (0, 0, 1, 1, 1, 0, -1, -1, -1)
WEIGHT = tuple(4 / 9 if c == 0 else 1 / 9 if c == 1 else 1 / 36 for c in (x * x + y * y for x, y in zip(CX, CY)))
COMPUTE = {"f32": torch.float32, "f64": torch.float64, "f16": torch.float32, "bf16": torch.float32}
MOVING = {"f32": 4, "f64": 8, "f16": 2, "bf16": 2}


def film(name, shape, nx, ny, steps, dtype="f32", tau=1.0):
    return dict(name=name, kind="film", shape=shape, nx=nx, ny=ny, steps=steps, dtype=dtype, tau=tau)


def listed():
    return [
        # the smallest run: a hanging film's growth, its height read every 100 steps
        film("ripple_128", "ripple", 128, 128, 100),
        # a spreading drop off the default viscosity (the paper varies it over tau = 0.9, 1, 1.2)
        film("drop_512_tau", "drop", 512, 512, 100, tau=0.9),
        # a verification run in double precision on a ragged lattice
        film("noise_250_f64", "noise", 250, 190, 50, dtype="f64", tau=0.8),
        # dewetting on a lattice of odd width, in the L2 cache
        film("noise_509_odd", "noise", 509, 387, 100),
        # the headline workload, and the same with half-width populations
        film("noise_2048", "noise", 2048, 2048, 40),
        film("noise_2048_f16", "noise", 2048, 2048, 40, dtype="f16"),
        # a large dewetting run off the default viscosity, ragged
        film("noise_2000_tau", "noise", 2000, 1530, 40, tau=1.2),
        # sliding drops at many Bond numbers, advanced together
        dict(name="sweep_32", kind="sweep", domains=32, lo=256, hi=1024, steps=20, dtype="f32", tau=1.0),
        # one gradient of a film-shape loss, as an optimiser of the wettability pattern asks for
        dict(name="gradient_512", kind="gradient", nx=512, ny=512, steps=400, dtype="f32", tau=1.0),
        # a plot file's fields
        dict(name="readout_2048", kind="readout", nx=2048, ny=2048, dtype="f32", tau=1.0),
        # a checkpoint read and written
        dict(name="restart_1024", kind="restart", nx=1024, ny=1024, dtype="f32", tau=1.0),
        # the monitoring of a sweep: drop positions, velocities, wetted areas
        dict(name="diagnose_32", kind="diagnose", domains=32, lo=256, hi=1024, dtype="f32", tau=1.0),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["film"] * 6 + ["sweep", "gradient", "readout", "restart", "diagnose"])
    tau = rng.choice([1.0, 1.0, 1.0, 0.8, 0.9, 1.2])
    dtype = rng.choice(["f32", "f32", "f32", "f16", "bf16", "f64"])
    if kind in ("sweep", "diagnose"):
        c = dict(kind=kind, domains=rng.randint(4, 32), lo=rng.choice([128, 192, 256]), hi=rng.choice([512, 768, 1024]),
                 dtype="f32" if dtype == "f64" else dtype, tau=tau)
        return dict(c, steps=rng.randint(10, 20)) if kind == "sweep" else c
    if kind == "gradient":
        n = _size(rng, 128, 512)
        return dict(kind=kind, nx=n, ny=_size(rng, 128, 512), steps=rng.randint(100, 400), dtype="f32", tau=tau)
    if kind in ("readout", "restart"):
        return dict(kind=kind, nx=_size(rng, 256, 2048), ny=_size(rng, 256, 2048), dtype=dtype, tau=tau)
    hi = 512 if dtype == "f64" else 2048
    nx, ny = _size(rng, 100, hi), _size(rng, 100, hi)
    most = 50 * 512 * 512 if dtype == "f64" else 40 * 2048 * 2048
    steps = max(10, min(_size(rng, 20, 200), most // (nx * ny)))
    shape = rng.choice(["ripple", "drop", "noise", "noise"])
    return {k: v for k, v in film("", shape, nx, ny, steps, dtype, tau).items() if k != "name"}


# ------------------------------------------------------------------ inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(gen, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=gen, device="cuda", dtype=torch.float64)


def _away(n, c):
    """Periodic distance of 0 .. n-1 from c."""
    d = (torch.arange(n, device="cuda", dtype=torch.float64) - c).abs()
    return torch.minimum(d, n - d)


def _cap(nx, ny, cx, cy, rb, theta):
    """Spherical cap of base radius rb and contact angle theta on the precursor film."""
    rad, hd = rb / math.sin(theta), rb / math.sin(theta) * (1 - math.cos(theta))
    r2 = _away(nx, cx)[None, :] ** 2 + _away(ny, cy)[:, None] ** 2
    return ((rad * rad - r2).clamp_min(0.0).sqrt() - (rad - hd)).clamp_min(HSTAR)


def _striped(gen, nx, ny):
    """Stripes at 10 and 40 degrees plus 32 discs at 10 degrees, in radians."""
    period = max(2, min(256, nx))
    x = torch.arange(nx, device="cuda")
    th = torch.where(x % period < period // 2, 10.0, 40.0).double().expand(ny, nx).clone()
    scale = min(1.0, min(nx, ny) / 512.0)
    draws = _uniform(gen, 0.0, 1.0, 32, 3).tolist()
    for a, b, c in draws:
        r = (16.0 + 48.0 * c) * scale
        th[_away(nx, a * nx)[None, :] ** 2 + _away(ny, b * ny)[:, None] ** 2 <= r * r] = 10.0
    return torch.deg2rad(th)


def _film_inputs(case, seed):
    """(params, h0, theta or None) of a film case, in the precision that the run is given."""
    gen, nx, ny, dt = _generator(seed), case["nx"], case["ny"], COMPUTE[case["dtype"]]
    p = dict(BASE, nx=nx, ny=ny, tau=case["tau"])
    theta = None
    if case["shape"] == "ripple":
        p.update(g=-5e-5, delta=0.0, theta_uniform=0.0)
        phase, amp = _uniform(gen, 0.0, 2 * math.pi, 1), _uniform(gen, 1e-3, 2e-3, 1)
        x = torch.arange(nx, device="cuda", dtype=torch.float64)
        h0 = (1 + amp * torch.sin(2 * math.pi * x / nx + phase)).expand(ny, nx)
    elif case["shape"] == "drop":
        p.update(theta_uniform=math.radians(20.0))
        rb, cx, cy = (_uniform(gen, 0.0, 1.0, 3)).tolist()
        h0 = _cap(nx, ny, (0.4 + 0.2 * cx) * nx, (0.4 + 0.2 * cy) * ny, (0.2 + 0.05 * rb) * min(nx, ny), math.radians(19.0))
    else:
        h0 = 1 + _uniform(gen, -1e-2, 1e-2, ny, nx)
        theta = _striped(gen, nx, ny).to(dt)
    return p, h0.to(dt).contiguous(), theta


def _domain_inputs(case, seed):
    """The domains of a sweep: Lx a multiple of 64, Ly = Lx / 2, a drop under a tangential force set by its Bond number.
    The sizes come from the case, as a sweep's do; drops and forces from the seed."""
    gen, n, dt = _generator(seed), case["domains"], COMPUTE[case["dtype"]]
    th = math.radians(40.0)
    draws = _uniform(gen, 0.0, 1.0, n, 4).tolist()
    lo, hi = case["lo"] // 64, case["hi"] // 64
    out = []
    for i, (a, b, c, d) in enumerate(draws):
        lx = 64 * (lo + (i * 7 + i // 3) % (hi - lo + 1))
        ly = lx // 2
        rb = min(40.0 + 40.0 * a, 0.4 * ly)
        rad = rb / math.sin(th)
        vol = math.pi / 3 * rad ** 3 * (2 + math.cos(th)) * (1 - math.cos(th)) ** 2
        bond = 0.05 * 20.0 ** ((i + d) / n)
        gx = bond * BASE["gamma"] / (3 * vol / (4 * math.pi)) ** (2 / 3)
        h0 = _cap(lx, ly, (0.3 + 0.4 * b) * lx, (0.3 + 0.4 * c) * ly, rb, th)
        out.append((dict(BASE, nx=lx, ny=ly, tau=case["tau"], gx_body=gx, theta_uniform=th), h0.to(dt).contiguous()))
    return out


def _populations(gen, h):
    """Populations of a film of height h that moves and is off equilibrium, (9, ny, nx) in float64."""
    ny, nx = h.shape
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :] * (2 * math.pi / nx)
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None] * (2 * math.pi / ny)
    ph = _uniform(gen, 0.0, 2 * math.pi, 2).tolist()
    ux, uy = 1e-3 * torch.sin(x + ph[0]) * torch.cos(y), 6e-4 * torch.cos(2 * x) * torch.sin(y + ph[1])
    f = _equilibrium(h, h * ux, h * uy, 0.0)
    f[1:] += _uniform(gen, -1e-5, 1e-5, 8, ny, nx)
    return f


def _state_inputs(case, seed):
    """(params, h0, theta, populations) of a read-out or restart: a film in motion over a patterned substrate."""
    gen, nx, ny, dt = _generator(seed), case["nx"], case["ny"], COMPUTE[case["dtype"]]
    p = dict(BASE, nx=nx, ny=ny, tau=case["tau"], gx_body=1e-5)
    h = 1 + _uniform(gen, -5e-2, 5e-2, ny, nx)
    theta = _striped(gen, nx, ny).to(dt)
    return p, h.to(dt), theta, _populations(gen, h)


def _gradient_inputs(case, seed):
    gen, nx, ny, dt = _generator(seed), case["nx"], case["ny"], COMPUTE[case["dtype"]]
    p = dict(BASE, nx=nx, ny=ny, tau=case["tau"])
    h0 = 1 + _uniform(gen, -1e-2, 1e-2, ny, nx)
    theta = torch.deg2rad(30 + 5 * torch.randn(ny, nx, generator=gen, device="cuda", dtype=torch.float64))
    target = torch.zeros(ny, nx, device="cuda", dtype=torch.float64)
    for a, b, c in _uniform(gen, 0.0, 1.0, 8, 3).tolist():
        s = min(nx, ny) * (1 + c) / 64
        target += torch.exp(-(_away(nx, a * nx)[None, :] ** 2 + _away(ny, b * ny)[:, None] ** 2) / (2 * s * s))
    target *= h0.sum() / target.sum()
    return p, h0.to(dt), theta.to(dt), target.to(dt)


# --------------------------------------------------------------- the passes

def prepare(case, seed):
    kind, dtype = case["kind"], case["dtype"]
    if kind == "film":
        p, h0, theta = _film_inputs(case, seed)
        return dict(kind=kind, steps=case["steps"], sim=ThinFilm(p, h0, theta, dtype=dtype))
    if kind in ("sweep", "diagnose"):
        films = [ThinFilm(p, h0, None, dtype=dtype) for p, h0 in _domain_inputs(case, seed)]
        if kind == "diagnose":
            gen = _generator(seed + 1)
            for f in films:
                f.set_state(_populations(gen, f.h0_dev.double()))
        return dict(kind=kind, steps=case.get("steps", 0), films=films, batch=FilmBatch(films))
    if kind == "gradient":
        p, h0, theta, target = _gradient_inputs(case, seed)
        return dict(kind=kind, params=p, h0=h0.requires_grad_(), theta=theta.requires_grad_(), target=target,
                    steps=case["steps"], dtype=dtype)
    p, h0, theta, f = _state_inputs(case, seed)
    sim = ThinFilm(p, h0, theta, dtype=dtype)
    if kind == "readout":
        sim.set_state(f)
        return dict(kind=kind, sim=sim)
    return dict(kind=kind, sim=sim, saved=f)


def run(state):
    kind = state["kind"]
    if kind == "film":
        state["sim"].step(state["steps"])
        return state["sim"].h()
    if kind == "sweep":
        state["batch"].step(state["steps"])
        return [f.h() for f in state["films"]]
    if kind == "diagnose":
        return state["batch"].diagnostics(2 * HSTAR)
    if kind == "gradient":
        h = evolve(state["theta"], state["h0"], state["params"], state["steps"], state["dtype"])
        loss = 0.5 * ((h - state["target"]) ** 2).sum()
        gth, gh0 = torch.autograd.grad(loss, (state["theta"], state["h0"]))
        return dict(h=h, theta=gth, h0=gh0)
    if kind == "readout":
        return dict(state["sim"].moments(), **state["sim"].pressure_force())
    state["sim"].set_state(state["saved"])
    return state["sim"].get_state()


def work(case):
    """One pass: the state and the substrate read once, the state and what is asked for written once; about 200 operations a
    node and step (moments 25, pressure 30, force 45, equilibria and collision 100), three times that for an adjoint step."""
    nodes = sum(p["nx"] * p["ny"] for p in _shapes(case)) if "domains" in case else case["nx"] * case["ny"]
    wide = 8 if case["dtype"] == "f64" else 4
    state, steps, kind = wide + 8 * MOVING[case["dtype"]], case.get("steps", 0), case["kind"]
    if kind == "film":
        kappa = wide if case["shape"] == "noise" else 0
        return dict(bytes=nodes * (2 * state + kappa + wide), flops=200 * nodes * steps)
    if kind == "sweep":
        return dict(bytes=nodes * (2 * state + wide), flops=200 * nodes * steps)
    if kind == "gradient":  # h0, theta and target in, h and two gradients out; forward once, adjoint once
        return dict(bytes=nodes * 6 * wide, flops=800 * nodes * steps)
    if kind == "readout":
        return dict(bytes=nodes * (state + wide + 6 * wide), flops=100 * nodes)
    if kind == "diagnose":
        return dict(bytes=nodes * state, flops=60 * nodes)
    return dict(bytes=nodes * (2 * 72 + 2 * state), flops=18 * nodes)


def _shapes(case):
    lo, hi = case["lo"] // 64, case["hi"] // 64
    for i in range(case["domains"]):
        lx = 64 * (lo + (i * 7 + i // 3) % (hi - lo + 1))
        yield dict(nx=lx, ny=lx // 2)


# ------------------------------------------- the same results in 64 bits

def _equilibrium(h, jx, jy, g):
    j2, f = jx * jx + jy * jy, []
    for l in range(9):
        if l == 0:
            f.append(h - 5 * g * h * h / 6 - 2 * j2 / (3 * h))
        else:
            cj, s = CX[l] * jx + CY[l] * jy, 1.0 if l % 2 else 0.25
            f.append(s * (g * h * h / 6 + cj / 3 + cj * cj / (2 * h) - j2 / (6 * h)))
    return torch.stack(f)


def _gradient(a):
    e, w = torch.roll(a, -1, 1), torch.roll(a, 1, 1)
    n, s = torch.roll(a, -1, 0), torch.roll(a, 1, 0)
    ne, nw, se, sw = torch.roll(n, -1, 1), torch.roll(n, 1, 1), torch.roll(s, -1, 1), torch.roll(s, 1, 1)
    return (e - w) / 3 + (ne - nw + se - sw) / 12, (n - s) / 3 + (ne - se + nw - sw) / 12


def _laplacian(a):
    n, s = torch.roll(a, -1, 0), torch.roll(a, 1, 0)
    diag = torch.roll(n, -1, 1) + torch.roll(n, 1, 1) + torch.roll(s, -1, 1) + torch.roll(s, 1, 1)
    return (4 * (torch.roll(a, -1, 1) + torch.roll(a, 1, 1) + n + s) + diag - 20 * a) / 6


def _kappa(p, theta):
    c = (p["n_exp"] - 1) * (p["m_exp"] - 1) / ((p["n_exp"] - p["m_exp"]) * p["hstar"])
    return (1 - torch.cos(theta)) * c


def _moments(f):
    return f.sum(0), f[1] + f[2] + f[8] - f[4] - f[5] - f[6], f[2] + f[3] + f[4] - f[6] - f[7] - f[8]


def _pressure_force(p, kappa, f):
    h, jx, jy = _moments(f)
    r = p["hstar"] / h
    pr = -p["gamma"] * (_laplacian(h) + p["pi_sign"] * kappa * (r ** p["n_exp"] - r ** p["m_exp"]))
    gx, gy = _gradient(pr)
    fric = 2 * (p["tau"] - 0.5) / (2 * h * h + 6 * p["delta"] * h + 3 * p["delta"] ** 2)
    return h, jx, jy, pr, h * (p["gx_body"] - gx) - fric * jx, h * (p["gy_body"] - gy) - fric * jy


def _step(p, kappa, f):
    h, jx, jy, _, fx, fy = _pressure_force(p, kappa, f)
    om, eq = 1 / p["tau"], _equilibrium(h, jx, jy, p["g"])
    out = [(1 - om) * f[l] + om * eq[l] + 3 * WEIGHT[l] * (CX[l] * fx + CY[l] * fy) for l in range(9)]
    return torch.stack([torch.roll(o, (CY[l], CX[l]), (0, 1)) for l, o in enumerate(out)])


def _run(p, kappa, h0, steps):
    zero = torch.zeros_like(h0)
    f = _equilibrium(h0, zero, zero, p["g"])
    for _ in range(steps):
        f = _step(p, kappa, f)
    return f.sum(0)


def _uniform_kappa(p):
    return _kappa(p, torch.tensor(p.get("theta_uniform", 0.0), device="cuda", dtype=torch.float64))


def exact(case, seed):
    kind = case["kind"]
    if kind == "film":
        p, h0, theta = _film_inputs(case, seed)
        return _run(p, _uniform_kappa(p) if theta is None else _kappa(p, theta.double()), h0.double(), case["steps"])
    if kind == "sweep":
        return [_run(p, _uniform_kappa(p), h0.double(), case["steps"]) for p, h0 in _domain_inputs(case, seed)]
    if kind == "diagnose":
        gen, rows = _generator(seed + 1), []
        for p, h0 in _domain_inputs(case, seed):
            h, jx, jy = _moments(_populations(gen, h0.double()))
            wet = (h > 2 * HSTAR).double()
            ax = torch.arange(p["nx"], device="cuda", dtype=torch.float64)[None, :] * (2 * math.pi / p["nx"])
            ay = torch.arange(p["ny"], device="cuda", dtype=torch.float64)[:, None] * (2 * math.pi / p["ny"])
            hw = h * wet
            rows.append(torch.stack([h.sum(), hw.sum(), (wet * jx).sum(), (wet * jy).sum(), wet.sum(), h.max(),
                                     (hw * ax.cos()).sum(), (hw * ax.sin()).sum(), (hw * ay.cos()).sum(),
                                     (hw * ay.sin()).sum(), (h * ax.cos()).sum(), (h * ax.sin()).sum()]))
        return torch.stack(rows)
    if kind == "gradient":
        from torch.utils.checkpoint import checkpoint
        p, h0, theta, target = _gradient_inputs(case, seed)
        h0, theta, target = h0.double().requires_grad_(), theta.double().requires_grad_(), target.double()
        kappa, zero, left = _kappa(p, theta), torch.zeros_like(h0), case["steps"]
        f = _equilibrium(h0, zero, zero, p["g"])

        def some(f, kappa, n):
            for _ in range(n):
                f = _step(p, kappa, f)
            return f
        while left:
            n = min(20, left)
            f, left = checkpoint(some, f, kappa, n, use_reentrant=False), left - n
        h = f.sum(0)
        gth, gh0 = torch.autograd.grad(0.5 * ((h - target) ** 2).sum(), (theta, h0))
        return dict(h=h.detach(), theta=gth, h0=gh0)
    p, _, theta, f = _state_inputs(case, seed)
    if kind == "restart":
        return f
    h, jx, jy, pr, fx, fy = _pressure_force(p, _kappa(p, theta.double()), f)
    return dict(h=h, ux=jx / h, uy=jy / h, p=pr, fx=fx, fy=fy)
