"""Measured cases of the D2Q9 KBC library: what a simulation program has it do.

A case is one of five kinds of work, each through the package's public entry
points:

* ``run``      a fresh field is handed over (``Lattice.init``), advanced
               (``Lattice.step``) and read back (``Lattice.moments``);
* ``restart``  a checkpoint is loaded (``Lattice.set_populations``), advanced
               and written out again (``Lattice.populations``);
* ``history``  a field is advanced and sampled: ``Lattice.diagnostics``,
               ``Lattice.diagnostics_ext``, as ``runs.history`` does;
* ``slabs``    the grid is split into y-slabs that exchange halos before every
               step (``slabs.SlabGroup``);
* ``spectrum`` shell-averaged energy and enstrophy spectra of a velocity field;
* ``adjoint``  an objective of the final field and its gradients through
               ``autograd.kbc_objective`` and ``backward``.

The flows are random solenoidal velocity fields carried by a uniform drift
(the decaying-turbulence family), doubly periodic shear layers and
Taylor-Green vortices, all periodic on any nx x ny grid; the seed moves their
phases and amplitudes.
"""
from __future__ import annotations

import math

import torch

from paper_1507_02509_gb300 import Lattice, VARIANTS
from paper_1507_02509_gb300.autograd import kbc_objective
from paper_1507_02509_gb300.slabs import SlabGroup
from paper_1507_02509_gb300.spectra import energy_spectrum, shell_count

# stored bytes per population
ELEMENT = {"f64": 8, "f32": 4, "f16": 2}
# floating-point operations of one node update (moments, equilibrium, split,
# entropic products, update; fused multiply-adds count twice)
STEP_FLOPS = {"lbgk": 110, "A": 300, "B": 290, "C": 270, "D": 265}


def _case(name, kind, nx, ny, variant, dtype, steps, flow="turbulence", beta=0.99, gamma="entropic",
          parts=1, every=0, objective="ke"):
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "variant": variant, "dtype": dtype,
            "steps": steps, "flow": flow, "beta": beta, "gamma": gamma, "parts": parts,
            "every": every, "objective": objective}


def listed():
    return [
        # the FP64 validation run: the 64^2 Taylor-Green vortex, 1000 steps
        _case("vortex-64-f64", "run", 64, 64, "B", "f64", 1000, "vortex", 1.0 / 1.06),
        # the smallest call: a coupled or interactive program takes a few steps
        # of a small grid and looks at the fields again
        _case("vortex-128-f32", "run", 128, 128, "C", "f32", 10, "vortex", 1.0 / 1.06),
        # the doubly periodic shear layer in working precision
        _case("shear-1024-f32", "run", 1024, 1024, "B", "f32", 200, "shear", 0.9918),
        # the same layer in double, against which the others are validated
        _case("shear-1024-f64", "run", 1024, 1024, "B", "f64", 40, "shear", 0.9918),
        # under-resolved decaying turbulence with half-precision storage
        _case("turbulence-4096-f16", "run", 4096, 4096, "B", "f16", 100, "turbulence", 0.99268),
        # the throughput run: the largest grid, 19 GB of populations
        _case("turbulence-16384-f32", "run", 16384, 16384, "B", "f32", 50, "turbulence", 0.9985),
        # checkpoint and restart on a domain whose width is no multiple of a
        # vector or a warp
        _case("restart-1001x750-f32", "restart", 1001, 750, "D", "f32", 100, "turbulence", 0.98),
        # energy, enstrophy, stabiliser, palinstrophy and entropy histories
        _case("history-4096-f32", "history", 4096, 4096, "B", "f32", 100, "turbulence", 0.99268,
              every=50),
        # spectra of the turbulence figures
        _case("spectrum-4096", "spectrum", 4096, 4096, "B", "f64", 0),
        # one large grid as four y-slabs, plain LBGK for comparison with KBC
        _case("slabs-2048x1536-f32", "slabs", 2048, 1536, "lbgk", "f32", 20, parts=4, beta=0.99),
        # gradient of the final kinetic energy with respect to the initial
        # velocity and beta, checkpoints every 100 steps
        _case("adjoint-512-f32", "adjoint", 512, 512, "B", "f32", 100, "turbulence", 0.982,
              every=100),
        # gradient of a field misfit in double, several segments recomputed
        _case("adjoint-200-f64", "adjoint", 200, 200, "C", "f64", 60, "turbulence", 0.97,
              every=20, objective="misfit"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extent(rng, lo, hi):
    """A grid extent spread over [lo, hi] by its logarithm: half of them
    multiples of 128 or 32 where that fits, the others as they come."""
    n = _log_int(rng, lo, hi)
    m = rng.choice((1, 1, 32, 128))
    return max(lo, n // m * m) if n >= m else n


def draw(rng):
    kind = rng.choice(("run", "run", "run", "restart", "history", "slabs", "spectrum", "adjoint"))
    dtype = rng.choice(("f64", "f32", "f32", "f16"))
    variant = rng.choice(("lbgk", "A", "B", "B", "C", "D"))
    flow = rng.choice(("turbulence", "turbulence", "shear", "vortex"))
    beta = round(rng.uniform(0.9, 0.998), 4)
    gamma = "entropic" if rng.random() < 0.85 else "regularised"
    if kind == "spectrum":
        n = 2 * _log_int(rng, 32, 3000)
        return _case("", kind, n, n, "B", "f64", 0)
    if kind == "adjoint":
        nx, ny = _extent(rng, 32, 700), _extent(rng, 32, 700)
        steps = _log_int(rng, 5, 60)
        return _case("", kind, nx, ny, variant, rng.choice(("f64", "f32")), steps, "turbulence", beta,
                     gamma, every=rng.choice((5, 10, 20, 100)), objective=rng.choice(("ke", "misfit")))
    nx, ny = _extent(rng, 32, 5000), _extent(rng, 32, 5000)
    # between 1 and 300 steps, at most 2e9 node updates (a quarter of that in double)
    most = (5e8 if dtype == "f64" else 2e9) / (nx * ny)
    steps = _log_int(rng, 1, max(2, min(300, int(most))))
    if kind == "history":
        return _case("", kind, nx, ny, variant, dtype, steps, flow, beta, gamma,
                     every=max(1, steps // rng.choice((1, 2, 3))))
    parts = min(rng.choice((2, 3, 4, 8)), ny) if kind == "slabs" else 1
    return _case("", kind, nx, ny, variant, dtype, steps, flow, beta, gamma, parts=parts)


# ------------------------------------------------------------------ inputs


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _turbulence(nx, ny, k0, urms, g):
    """Solenoidal random velocity, E(k) ~ k^4 exp(-2 (k/k0)^2), rms speed urms,
    on any periodic grid (k in cycles per longer side)."""
    n = max(nx, ny)
    ky = torch.fft.fftfreq(ny, 1.0 / ny, dtype=torch.float64, device="cuda")[:, None] * (n / ny)
    kx = torch.fft.rfftfreq(nx, 1.0 / nx, dtype=torch.float64, device="cuda")[None, :] * (n / nx)
    k2 = kx * kx + ky * ky
    # white noise has as much energy per mode everywhere: psi's amplitude is sqrt(E / k) / k
    noise = torch.fft.rfft2(torch.randn(ny, nx, dtype=torch.float64, device="cuda", generator=g))
    noise *= k2.pow(0.25) * torch.exp(-k2 / (k0 * k0))
    out = []
    for c in (1j * ky, -1j * kx):
        out.append(torch.fft.irfft2(noise * c, s=(ny, nx)))
    ux, uy = out
    s = urms / float(torch.sqrt((ux * ux + uy * uy).mean()))
    return ux.mul_(s), uy.mul_(s)


def _fields(case, seed):
    """rho, ux, uy of a case, float64 on the GPU."""
    nx, ny = case["nx"], case["ny"]
    g = _generator(seed)
    a = torch.rand(4, generator=g, device="cuda", dtype=torch.float64).cpu().tolist()
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :] / nx + a[0]
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None] / ny + a[1]
    u0 = 0.035 + 0.01 * a[2]
    if case["flow"] == "vortex":
        ux = -u0 * torch.cos(2 * math.pi * x) * torch.sin(2 * math.pi * y)
        uy = u0 * torch.sin(2 * math.pi * x) * torch.cos(2 * math.pi * y)
    elif case["flow"] == "shear":
        yy = torch.remainder(y, 1.0)
        ux = torch.where(yy <= 0.5, u0 * torch.tanh(80 * (yy - 0.25)), u0 * torch.tanh(80 * (0.75 - yy)))
        ux = ux.expand(ny, nx)
        uy = (0.05 * u0 * torch.sin(2 * math.pi * (x + 0.25))).expand(ny, nx)
    else:
        k0 = min(16.0, max(nx, ny) / 16.0)
        ux, uy = _turbulence(nx, ny, k0, 0.03, g)
    # carried by a uniform drift, which leaves no conserved sum at zero
    ux = (ux + 0.004).contiguous()
    uy = (uy + 0.002).contiguous()
    return torch.ones(ny, nx, dtype=torch.float64, device="cuda"), ux, uy


def _gamma(case):
    return 1.0 / case["beta"] if case["gamma"] == "regularised" and case["variant"] != "lbgk" else None


def prepare(case, seed):
    kind = case["kind"]
    rho, ux, uy = _fields(case, seed)
    state = {"case": case, "rho": rho, "ux": ux, "uy": uy}
    if kind == "spectrum":
        return state
    if kind == "adjoint":
        # a program that works in double differentiates doubles, any other floats
        t = torch.float64 if case["dtype"] == "f64" else torch.float32
        state["u0"] = torch.stack((ux, uy)).to(t).requires_grad_()
        state["beta"] = torch.tensor(case["beta"], dtype=t, requires_grad=True)
        if case["objective"] == "misfit":
            state["target"] = torch.stack(_fields(case, seed + 7919)[1:])
        return state
    if kind == "slabs":
        state["group"] = SlabGroup(case["nx"], case["ny"], case["parts"], variant=case["variant"],
                                   beta=case["beta"], dtype=case["dtype"])
        lattices = state["group"].slabs
    else:
        state["lattice"] = Lattice(case["nx"], case["ny"], variant=case["variant"], beta=case["beta"],
                                   dtype=case["dtype"])
        lattices = [state["lattice"]]
    if _gamma(case) is not None:
        for lat in lattices:
            lat.set_gamma(_gamma(case))
    if kind == "restart":
        state["f"] = _equilibrium(rho, ux, uy) + _weights(rho)
        # a checkpoint is not in equilibrium
        g = _generator(seed + 1)
        state["f"] *= 1.0 + 1e-3 * torch.randn(state["f"].shape, dtype=torch.float64, device="cuda", generator=g)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "run":
        return state["lattice"].init(state["rho"], state["ux"], state["uy"]).step(case["steps"]).moments()
    if kind == "restart":
        lat = state["lattice"]
        lat.set_populations(state["f"])
        return lat.step(case["steps"]).populations()
    if kind == "history":
        lat = state["lattice"].init(state["rho"], state["ux"], state["uy"])
        samples, done = [], 0
        while done < case["steps"]:
            k = min(case["every"], case["steps"] - done)
            lat.step(k)
            lat.sync()
            done += k
            samples.append({**lat.diagnostics(), **lat.diagnostics_ext()})
        return samples
    if kind == "slabs":
        return state["group"].init(state["rho"], state["ux"], state["uy"]).step(case["steps"]).moments()
    if kind == "spectrum":
        return energy_spectrum(state["ux"], state["uy"])
    u0, beta = state["u0"], state["beta"]
    u0.grad = beta.grad = None
    J = kbc_objective(u0, beta, rho0=state["rho"], variant=case["variant"], dtype=case["dtype"],
                      steps=case["steps"], ckpt_every=case["every"], objective=case["objective"],
                      u_target=state.get("target"), gamma_fixed=_gamma(case))
    J.backward()
    return {"J": J.detach(), "du0": u0.grad, "dbeta": beta.grad}


def work(case):
    """Each field in and out once; each step reads and writes the nine
    populations once."""
    n = case["nx"] * case["ny"]
    kind, steps = case["kind"], case["steps"]
    pops = 9 * ELEMENT[case["dtype"]]
    flops = STEP_FLOPS[case["variant"]]
    if kind in ("run", "slabs"):
        return {"bytes": n * (48 + 2 * pops * steps), "flops": n * flops * steps}
    if kind == "restart":
        return {"bytes": n * (144 + 2 * pops * steps), "flops": n * flops * steps}
    if kind == "history":
        samples = -(-steps // case["every"])
        return {"bytes": n * (24 + 2 * pops * steps + 2 * pops * samples),
                "flops": n * (flops * steps + samples * (flops + 400))}
    if kind == "spectrum":
        return {"bytes": n * 16, "flops": 2 * 2.5 * n * math.log2(n)}
    # adjoint: one forward sweep, one reverse sweep of about three times its arithmetic
    real = 9 * (8 if case["dtype"] == "f64" else 4)
    u0 = 8 if case["dtype"] == "f64" else 4
    return {"bytes": n * (8 + 4 * u0 + steps * (2 * pops + pops + 2 * real)), "flops": n * flops * 4 * steps}


# ------------------------------------------------------------------ 64-bit values

# v_i = (a, b), i = 3 (b + 1) + (a + 1)
_A = [i % 3 - 1 for i in range(9)]
_B = [i // 3 - 1 for i in range(9)]
_W = [(2.0 / 3.0 if a == 0 else 1.0 / 6.0) * (2.0 / 3.0 if b == 0 else 1.0 / 6.0) for a, b in zip(_A, _B)]


def _weights(like):
    return torch.tensor(_W, dtype=torch.float64, device=like.device)[:, None, None]


def _poly(ux, uy):
    """f^eq_i / (W_i rho) - 1."""
    uu = 1.5 * (ux * ux + uy * uy)
    xi = [a * ux + b * uy for a, b in zip(_A, _B)]
    return [x * (3.0 + 4.5 * x) - uu for x in xi]


def _equilibrium(rho, ux, uy):
    """f^eq - W."""
    return torch.stack([w * ((rho - 1.0) + rho * p) for w, p in zip(_W, _poly(ux, uy))])


def _macro(d):
    drho = d.sum(0)
    rho = 1.0 + drho
    jx = (d[2] - d[0]) + (d[8] - d[6]) + (d[5] - d[3])
    jy = (d[6] - d[0]) + (d[8] - d[2]) + (d[7] - d[1])
    return rho, drho, jx / rho, jy / rho


def _step(d, variant, beta, gamma):
    """One pull and collision of the deviations d_i = f_i - W_i; also gamma."""
    d = [torch.roll(d[i], (_B[i], _A[i]), (0, 1)) for i in range(9)]
    rho, drho, ux, uy = _macro(torch.stack(d))
    poly = _poly(ux, uy)
    df = [d[i] - _W[i] * (drho + rho * poly[i]) for i in range(9)]
    if variant == "lbgk":
        return torch.stack([d[i] - 2.0 * beta * df[i] for i in range(9)]), torch.full_like(rho, 2.0)
    corner = (df[0] + df[8]) + (df[2] + df[6])
    m20 = corner + (df[3] + df[5])
    m02 = corner + (df[1] + df[7])
    m11 = (df[0] + df[8]) - (df[2] + df[6])
    c20, c02 = (m20, m02) if variant in "AC" else (0.5 * (m20 - m02), 0.5 * (m02 - m20))
    cx, cy = (ux, uy) if variant in "AB" else (torch.zeros_like(ux), torch.zeros_like(uy))
    e0 = [lambda c: 0.5 * c * (c - 1.0), lambda c: 1.0 - c * c, lambda c: 0.5 * c * (c + 1.0)]
    e1 = [lambda c: c - 0.5, lambda c: -2.0 * c, lambda c: c + 0.5]
    e2 = [0.5, -1.0, 0.5]
    ds = [c20 * e2[a + 1] * e0[b + 1](cy) + c02 * e0[a + 1](cx) * e2[b + 1] + m11 * e1[a + 1](cx) * e1[b + 1](cy)
          for a, b in zip(_A, _B)]
    dh = [df[i] - ds[i] for i in range(9)]
    if gamma is None:
        inv = [1.0 / (_W[i] * (1.0 + poly[i])) for i in range(9)]
        sh = sum(ds[i] * dh[i] * inv[i] for i in range(9))
        hh = sum(dh[i] * dh[i] * inv[i] for i in range(9))
        some = hh > 0
        gam = torch.where(some, 1.0 / beta - (2.0 - 1.0 / beta) * sh / torch.where(some, hh, torch.ones_like(hh)),
                          torch.full_like(hh, 2.0))
    else:
        gam = torch.full_like(rho, gamma)
    return torch.stack([d[i] - beta * (2.0 * ds[i] + gam * dh[i]) for i in range(9)]), gam


def _diagnostics(d):
    rho, _, ux, uy = _macro(d)

    def dx(q):
        return 0.5 * (torch.roll(q, -1, 1) - torch.roll(q, 1, 1))

    def dy(q):
        return 0.5 * (torch.roll(q, -1, 0) - torch.roll(q, 1, 0))

    ke = 0.5 * (ux * ux + uy * uy)
    w = dx(uy) - dy(ux)
    zz = 0.5 * w * w
    pp = 0.5 * (dx(w) ** 2 + dy(w) ** 2)
    se = -sum((_W[i] + d[i]) * torch.log1p(d[i] / _W[i]) for i in range(9))

    def std(q):
        return float(torch.sqrt(((q - q.mean()) ** 2).mean()))

    return {"mass": float(rho.sum()), "px": float((rho * ux).sum()), "py": float((rho * uy).sum()),
            "E": float(ke.mean()), "Z": float(zz.mean()), "E_std": std(ke), "Z_std": std(zz),
            "P": float(pp.mean()), "P_std": std(pp), "S": float(se.mean()), "S_std": std(se)}


def exact(case, seed):
    kind, steps, beta = case["kind"], case["steps"], case["beta"]
    variant, gamma = case["variant"], _gamma(case)
    n = case["nx"] * case["ny"]
    if n * steps > 3e9:
        return None
    if kind == "adjoint":
        return _exact_adjoint(case, seed)
    rho, ux, uy = _fields(case, seed)
    if kind == "spectrum":
        return _exact_spectrum(ux, uy)
    if kind == "restart":
        d = prepare(case, seed)["f"] - _weights(rho)
    else:
        d = _equilibrium(rho, ux, uy)
    if kind == "history":
        samples, done = [], 0
        while done < steps:
            k = min(case["every"], steps - done)
            for _ in range(k):
                d, _g = _step(d, variant, beta, gamma)
            done += k
            # the stabiliser's statistics are those of badly conditioned
            # quotients, and gradients of half-precision fields are their
            # rounding noise: no values for them
            s = {key: None for key in ("gamma_mean", "gamma_min", "gamma_max")}
            s.update(_diagnostics(d))
            if case["dtype"] == "f16":
                s.update({key: None for key in ("P", "P_std", "Z", "Z_std", "S", "S_std")})
            samples.append(s)
        return samples
    for _ in range(steps):
        d, _g = _step(d, variant, beta, gamma)
    if kind == "restart":
        return d + _weights(rho)
    r, _, vx, vy = _macro(d)
    return r, vx, vy


def _exact_spectrum(ux, uy):
    n = ux.shape[-1]
    ky = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")[:, None]
    kx = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")[None, :]
    shell = torch.round(torch.sqrt(kx * kx + ky * ky)).long().reshape(-1)
    nb = shell_count(n)
    E = torch.zeros(nb, dtype=torch.float64, device="cuda")
    for u in (ux, uy):
        h = torch.fft.fft2(u) / (n * n)
        e = 0.5 * (h.real ** 2 + h.imag ** 2).reshape(-1)
        E += torch.bincount(shell, weights=e, minlength=nb)[:nb]
    k = torch.arange(nb, dtype=torch.float64, device="cuda")
    return k, E, (2 * math.pi * k / n) ** 2 * E


def _exact_adjoint(case, seed):
    """Reverse mode of the plain 64-bit steps, in stretches of ten."""
    from torch.utils.checkpoint import checkpoint

    state = prepare(case, seed)
    rho = state["rho"]
    u = state["u0"].detach().to(torch.float64).requires_grad_()
    b = torch.tensor(float(state["beta"].detach()), dtype=torch.float64, device="cuda", requires_grad=True)
    # the regularised mode holds its gamma while beta varies
    gamma = _gamma(case)

    def stretch(d, b, k):
        for _ in range(k):
            d, _g = _step(d, case["variant"], b, gamma)
        return d

    d = _equilibrium(rho, u[0], u[1])
    left = case["steps"]
    while left > 0:
        k = min(10, left)
        d = checkpoint(stretch, d, b, k, use_reentrant=False)
        left -= k
    r, _, ux, uy = _macro(d)
    if case["objective"] == "ke":
        J = (0.5 * r * (ux * ux + uy * uy)).sum()
    else:
        t = state["target"]
        J = 0.5 * ((ux - t[0]) ** 2 + (uy - t[1]) ** 2).sum()
    J.backward()
    return {"J": J.detach(), "du0": u.grad, "dbeta": b.grad}
