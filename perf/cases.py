"""Workloads of the split 6D Vlasov solver, through its public entry points.

A case is one call that a program of this library makes over and over: an Eq. (5) step
(FP32, FP64, BF16 or FP16 storage; self-consistent or with an external potential), a
drift of whole-cell shifts, the forward and backward of a differentiable run, the
velocity moments, the 16-bit codec.  Sizes are [nx, ny, nz] x [nux, nuy, nuz] cells.

    listed()              the named cases
    draw(rng)             one more case of the same ranges
    prepare(case, seed)   what a program holds before the call (inputs, context, fields)
    run(state)            one pass; returns its outputs, whole
    work(case)            bytes and operations a pass cannot do without
    tolerance(case)       how far another correct implementation may be off
    exact(case, seed)     the same outputs in 64 bits, as plain torch gives them
"""
import math
from fractions import Fraction

import numpy as np
import torch

from paper_2110_15867_gb300 import autograd, binding

DEV = "cuda"
DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
BOX = 1.0        # box side
A_HALF, A_FULL = 0.55, 0.56
FOUR_PI_G = 1.0
F_NU = 0.03      # neutrino fraction of the matter, which sets the background density


def _case(name, kind, n, nu, dtype, **more):
    c = {"name": name, "kind": kind, "dtype": dtype, "V": 8.0 if max(nu) >= 48 else 5.0}
    c.update(zip(("nx", "ny", "nz"), n))
    c.update(zip(("nux", "nuy", "nuz"), nu))
    c.update(more)
    return c


def listed():
    return [
        # the smallest run anyone makes (tests, convergence studies): launches and latency
        _case("step_f32_8x16", "step", (8, 8, 8), (16, 16, 16), "f32", sc=True),
        # FP64 storage, the parity and convergence mode, at the 16^3 x 16^3 parity size
        _case("step_f64_16x16", "step", (16, 16, 16), (16, 16, 16), "f64", sc=False),
        # an ordinary production step on a cube of 32^3 velocities
        _case("step_f32_32x32", "step", (32, 32, 32), (32, 32, 32), "f32", sc=True),
        # the largest: long position lines, f far larger than the cache
        _case("step_f32_64x32", "step", (64, 64, 32), (32, 32, 32), "f32", sc=True),
        # wide velocity cubes (|u| <= 8 u_T), the large self-consistent run's cube
        _case("step_f32_24x48", "step", (24, 24, 24), (48, 48, 48), "f32", sc=True),
        # sizes that no tile divides: non-cubic boxes, unequal velocity axes
        _case("step_f32_ragged", "step", (21, 26, 19), (24, 20, 28), "f32", sc=True),
        # 16-bit storage of f with a scale per line, both code types, both cube sizes
        _case("step_bf16_32x32", "step", (32, 32, 32), (32, 32, 32), "bf16", sc=True),
        _case("step_f16_24x48", "step", (24, 24, 24), (48, 48, 48), "f16", sc=False),
        # free streaming over a long step: Courant numbers up to 2.6, whole-cell shifts
        _case("drift_f32_shift", "drift", (32, 24, 32), (16, 16, 32), "f32", courant=2.6),
        # gradient of a density statistic with respect to the initial perturbation and the
        # potential, through a run with checkpoints
        _case("grad_f32_24x16", "grad", (24, 24, 24), (16, 16, 16), "f32", steps=2, every=1),
        # velocity moments of a snapshot: density, mean velocity, dispersion tensor
        _case("moments_f32_32x32", "moments", (32, 32, 24), (32, 32, 32), "f32"),
        # a snapshot into 16-bit storage and back
        _case("codec_bf16_24x32", "codec", (24, 24, 24), (32, 32, 32), "bf16"),
    ]


def draw(rng):
    kind = rng.choice(["step"] * 12 + ["drift", "grad", "grad", "moments", "codec"])
    dtype = {"drift": "f32", "grad": rng.choice(["f32"] * 3 + ["f64"]), "moments": "f32"}.get(kind) or (
        rng.choice(["bf16", "f16"]) if kind == "codec" else rng.choice(["f32"] * 6 + ["bf16", "bf16", "f16", "f64"]))
    coded = dtype in ("bf16", "f16")
    if kind == "grad":
        nu = (rng.choice([12, 16, 16, 16, 20, 24]),) * 3
    elif coded or rng.random() < 0.6:  # velocity cubes
        nu = (rng.choice([16, 32, 32, 48] if coded else [16, 16, 24, 32, 32, 40, 48]),) * 3
    else:
        nu = tuple(rng.choice(range(8, 49, 4)) for _ in range(3))
    most = {"grad": 5e6 if dtype == "f64" else 6e7, "drift": 5e8}.get(kind, 6e7 if dtype == "f64" else 1.5e9)
    while True:  # position lines from 6 to 64 cells, spread over their logarithm
        if rng.random() < 0.5:
            n = (rng.choice([8, 16, 24, 32, 48, 64]),) * 3
        else:
            n = tuple(int(round(math.exp(rng.uniform(math.log(6), math.log(64))))) for _ in range(3))
        if math.prod(n) * math.prod(nu) <= most:
            break
    c = _case("drawn", kind, n, nu, dtype)
    del c["name"]
    if kind == "step":
        c["sc"] = rng.random() < 0.7 and dtype != "f64"
    elif kind == "drift":
        c["courant"] = round(rng.uniform(1.2, 4.0), 2)
    elif kind == "grad":
        c["steps"], c["every"] = rng.choice([(1, 1), (2, 1), (2, 2)])
    return c


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

def _sizes(c):
    return (c["nx"], c["ny"], c["nz"]), (c["nux"], c["nuy"], c["nuz"])


def _modes(n):
    """Integer wave numbers of the three axes, broadcastable over n."""
    k = [torch.fft.fftfreq(m, 1.0 / m, dtype=torch.float64, device=DEV) for m in n]
    return k[0][:, None, None], k[1][None, :, None], k[2][None, None, :]


def _field(n, rms, g):
    """Gaussian random field with power spectrum ~ k^-2, zero mean, given rms (FP64)."""
    w = torch.randn(n, generator=g, dtype=torch.float64).to(DEV)
    kx, ky, kz = _modes(n)
    k = torch.sqrt(kx * kx + ky * ky + kz * kz)
    d = torch.fft.ifftn(torch.fft.fftn(w) / torch.where(k > 0, k, torch.full_like(k, math.inf))).real
    return d * (rms / d.std(correction=0))


def _centres(n, lo, hi):
    return lo + (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) * ((hi - lo) / n)


def _potential(n, g):
    """Eight seeded cosine modes of amplitude 0.1, wave numbers up to 3 (FP32)."""
    x = [_centres(m, 0.0, BOX) for m in n]
    phi = torch.zeros(n, dtype=torch.float64, device=DEV)
    for _ in range(8):
        k = torch.randint(-3, 4, (3,), generator=g).tolist()
        k = k if any(k) else [1, 0, 0]
        th = 2 * math.pi * float(torch.rand((), generator=g, dtype=torch.float64))
        phi += 0.1 * torch.cos(2 * math.pi * (k[0] * x[0][:, None, None] + k[1] * x[1][None, :, None] +
                                              k[2] * x[2][None, None, :]) / BOX + th)
    return phi.float()


def _poisson(rho, a):
    """nabla^2 phi = 4 pi G a^2 (rho - mean rho) on the periodic box, spectrally (FP64)."""
    kx, ky, kz = _modes(rho.shape)
    k2 = (2 * math.pi / BOX) ** 2 * (kx * kx + ky * ky + kz * kz)
    k2 = torch.where(k2 > 0, k2, torch.full_like(k2, math.inf))
    return torch.fft.ifftn(-FOUR_PI_G * a * a * torch.fft.fftn(rho) / k2).real


def _inputs(c, seed):
    """f0 = (1 + delta(x)) F(u - u_bulk), F the relativistic Fermi-Dirac shape, with the
    fields and the time step of a run: everything from the seed, f0 rounded to FP32 (FP64
    for FP64 storage)."""
    n, nu = _sizes(c)
    V = c["V"]
    g = torch.Generator().manual_seed(int(seed))
    delta = _field(n, 0.05, g)
    bulk = (torch.rand(3, generator=g, dtype=torch.float64) - 0.5).tolist()
    u = [_centres(m, -V, V) - b for m, b in zip(nu, bulk)]
    F = 1.0 / (torch.exp(torch.sqrt(u[0][:, None, None] ** 2 + u[1][None, :, None] ** 2 + u[2] ** 2)) + 1.0)
    dt64 = c["dtype"] == "f64"
    f = torch.empty(n + nu, dtype=torch.float64 if dt64 else torch.float32, device=DEV)
    for ix in range(n[0]):
        f[ix] = (1.0 + delta[ix])[:, :, None, None, None] * F
    rho = (1.0 + delta) * F.sum() * math.prod(2 * V / m for m in nu)
    bg = rho.mean() * (1.0 / F_NU - 1.0) * (1.0 + _field(n, 1.0, g))
    phi = _poisson(rho + bg, A_HALF - 0.01).float() if c.get("sc") else _potential(n, g)
    courant = c.get("courant") or 0.5 + 0.4 * float(torch.rand((), generator=g, dtype=torch.float64))
    dt = courant * A_HALF ** 2 * min(BOX / m / (V * (1 - 1.0 / k)) for m, k in zip(n, nu))
    # a velocity sweep's Courant number must stay below 1: the kicks take dt / 2
    top = max(float(_gradient(phi.double(), d).abs().max()) * nu[d] / (2 * V) for d in range(3))
    return {"f": f, "bg": bg, "phi": phi, "delta": delta.to(f.dtype), "F": F.to(f.dtype),
            "dt": min(dt, 1.6 / top) if c["kind"] in ("step", "grad") else dt}


def _initial(delta, F):
    return (1.0 + delta)[..., None, None, None] * F


def prepare(case, seed):
    c = dict(case)
    s = _inputs(c, seed)
    n, nu = _sizes(c)
    s["case"] = c
    if c["kind"] == "grad":
        s["run"] = autograd.Run(n + nu, dtype=DTYPES[c["dtype"]], device=DEV, L=BOX, V=c["V"])
        del s["f"]  # formed from delta in every pass
        s["delta"].requires_grad_(True)
        s["phi"].requires_grad_(True)
        kx, ky, kz = _modes(n)
        k = torch.sqrt(kx * kx + ky * ky + kz * kz)
        s["low"] = ((k > 0) & (k < 8)).double()
    elif c["kind"] == "codec":
        s["codes"] = torch.empty(n + nu, dtype=DTYPES[c["dtype"]], device=DEV)
        s["scale"] = torch.empty(n + nu[:2], dtype=torch.float32, device=DEV)
    else:
        scale = None
        if c["dtype"] in ("bf16", "f16"):
            s["f"], scale = binding.encode_lines(s["f"], DTYPES[c["dtype"]])
        s["v"] = binding.Vlasov(s["f"], L=BOX, V=c["V"], scale=scale)
        s["phi2"] = torch.empty_like(s["phi"])
        s["rho"] = torch.empty(n, dtype=torch.float64, device=DEV)
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "step":
        v, sc = s["v"], c["sc"]
        v.step(s["dt"], A_HALF, A_FULL, s["phi"], rho_bg=s["bg"] if sc else None, four_pi_G=FOUR_PI_G,
               phi_next=s["phi2"] if sc else None, rho_nu=s["rho"])
        out = {"f": v.f, "rho": s["rho"]}
        if v.scale is not None:
            out["scale"] = v.scale
        if sc:
            s["phi"], s["phi2"] = s["phi2"], s["phi"]  # the next step starts from the new potential
            out["phi"] = s["phi"]
        return out
    if kind == "drift":
        for axis in ("z", "y", "x"):
            s["v"].sweep(axis, s["dt"], A_HALF)
        return {"f": s["f"]}
    if kind == "grad":
        f0 = _initial(s["delta"], s["F"])
        rho = autograd.run_rho(f0, s["phi"], s["run"], s["dt"], A_HALF, c["steps"], c["every"])
        loss = (torch.fft.fftn(rho).abs() ** 2 * s["low"]).sum()
        ddelta, dphi = torch.autograd.grad(loss, (s["delta"], s["phi"]))
        return {"rho": rho.detach(), "ddelta": ddelta, "dphi": dphi}
    if kind == "moments":
        rho, umean, sigma2 = s["v"].moments()
        return {"rho": rho, "umean": umean, "sigma2": sigma2}
    codes, scale = binding.encode_lines(s["f"], s["codes"].dtype, codes=s["codes"], scale=s["scale"])
    return {"codes": codes, "scale": scale, "f": binding.decode_lines(codes, scale, torch.float32)}


# ----------------------------------------------------------------------------
# the least a pass needs, and how far another implementation may be off
# ----------------------------------------------------------------------------

def work(case):
    """Bytes: a kick stays inside a velocity cube and the three sweeps of a drift couple
    all of space, so a step reads and writes f once per kick and once per drift sweep.
    Operations: about 40 per cell and sweep (the flux, the limiter, the update), three
    times that for an adjoint sweep."""
    n, nu = _sizes(case)
    cells, lines = math.prod(n) * math.prod(nu), math.prod(n) * nu[0] * nu[1]
    es = {"f64": 8, "f32": 4}.get(case["dtype"], 2)
    f_bytes = cells * es + (lines * 4 if es == 2 else 0)
    kind = case["kind"]
    if kind == "step":
        return {"bytes": 5 * 2 * f_bytes, "flops": 9 * 40 * cells}
    if kind == "drift":
        return {"bytes": 3 * 2 * f_bytes, "flops": 3 * 40 * cells}
    if kind == "grad":
        # forward: nine sweeps, each read and written (the backward needs every sweep's
        # input); backward: input and lambda read, lambda written per sweep
        return {"bytes": case["steps"] * 9 * 5 * f_bytes, "flops": case["steps"] * 9 * 160 * cells}
    if kind == "moments":
        return {"bytes": f_bytes, "flops": 20 * cells}
    return {"bytes": cells * (4 + 2 + 2 + 4) + lines * 8, "flops": 4 * cells}


def tolerance(case):
    """Four times the distance from 64 bits seen at these sizes (FP32 sums rounded once per
    cell and sweep; 16-bit codes rounded stochastically once or more per sweep; in the FP32
    gradient a limiter branch that flips within rounding moves single cells by much, their
    sums over velocity by up to 2e-3).  The codec's results are defined to the bit."""
    if case["kind"] == "codec":
        return "exact"
    if case["kind"] == "grad":
        return {"rel": 1e-9, "max": 1e-7} if case["dtype"] == "f64" else {"rel": 0.01, "max": 0.3}
    if case["kind"] == "moments":
        return {"rel": 1e-6, "max": 1e-5}
    return {"f64": {"rel": 1e-14, "max": 1e-12}, "f32": {"rel": 4e-7, "max": 2e-5},
            "bf16": {"rel": 2e-2, "max": 0.5}, "f16": {"rel": 4e-3, "max": 0.1}}[case["dtype"]]


# ----------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ----------------------------------------------------------------------------

def _weight_powers():
    """K[p][m]: the mean over the departure interval [-s, 0] (cell units, the downwind face
    of the donor at 0) of the quintic through the primitive at the faces -3..2 is
    sum_m sum_p K[p][m] s^p c_m over the cells c_{j-2} .. c_{j+2}."""
    faces = [Fraction(k) for k in range(-3, 3)]
    K = [[Fraction(0)] * 5 for _ in range(5)]
    for q in range(1, 6):  # Lagrange basis polynomial of face q, powers of x
        poly = [Fraction(1)]
        for r in range(6):
            if r != q:
                d = faces[q] - faces[r]
                poly = [(poly[i - 1] if i else 0) / d - (faces[r] * poly[i] / d if i < len(poly) else 0)
                        for i in range(len(poly) + 1)]
        for p in range(1, 6):  # (P(0) - P(-s)) / s: -(-1)^p poly[p] s^(p-1)
            for m in range(q):  # the primitive at face q is the sum of the cells before it
                K[p - 1][m] += -((-1) ** p) * poly[p]
    return [[float(x) for x in row] for row in K]


_K = _weight_powers()


def _minmod4(a, b, c, d):
    lo = torch.minimum(torch.minimum(a, b), torch.minimum(c, d))
    hi = torch.maximum(torch.maximum(a, b), torch.maximum(c, d))
    return lo.clamp(min=0.0) + hi.clamp(max=0.0)


def _advect(c, nu, periodic):
    """Lines along dim 0 of c (flow toward +index): conservative semi-Lagrangian update by
    the Courant number nu >= 0 (broadcastable over c[0]) with the monotonicity constraint
    of Suresh & Huynh and the positivity clamp."""
    n = c.shape[0]
    s = nu - torch.floor(nu)
    if periodic:
        e = torch.cat([c[-3:], c, c[:2]])
    else:
        z = torch.zeros_like(c[:1])
        e = torch.cat([z, z, z, c, z, z])
    d = e[:-2] - 2 * e[1:-1] + e[2:]             # curvature of ext cells 1 ..
    m4 = _minmod4(4 * d[:-1] - d[1:], 4 * d[1:] - d[:-1], d[:-1], d[1:])  # face after ext cell 1 ..
    cm2, cm1, c0, cp1, cp2 = (e[k:k + n + 1] for k in range(5))
    up, dn = m4[:n + 1], m4[1:n + 2]
    w = [sum(_K[p][m] * s ** p for p in range(5)) for m in range(5)]
    fbar = w[0] * cm2 + w[1] * cm1 + w[2] * c0 + w[3] * cp1 + w[4] * cp2
    alpha = ((1 - s) / s.clamp(min=1e-300)).clamp(max=1e6)
    ful = c0 + alpha * (c0 - cm1)
    fmd = 0.5 * (c0 + cp1 - dn)
    flc = c0 + 0.5 * (c0 - cm1) + 4.0 / 3.0 * up
    lo = torch.maximum(torch.minimum(torch.minimum(c0, cp1), fmd), torch.minimum(torch.minimum(c0, ful), flc))
    hi = torch.minimum(torch.maximum(torch.maximum(c0, cp1), fmd), torch.maximum(torch.maximum(c0, ful), flc))
    F = torch.minimum((s * torch.minimum(torch.maximum(fbar, lo), hi)).clamp(min=0.0), c0)
    if not periodic:
        F = torch.cat([torch.zeros_like(F[:1]), F[1:-1], torch.zeros_like(F[:1])])
    return c + (F[:-1] - F[1:])


def _chunks(n_rows, row_cells):
    step = max(1, int(2 ** 25 // row_cells))
    return [(i, min(n_rows, i + step)) for i in range(0, n_rows, step)]


def _position(f, ax, c, dt):
    """D_ax of Eq. (3) in place (FP64)."""
    n, nu = _sizes(c)
    V = c["V"]
    dx = BOX / n[ax]
    for j in range(nu[ax]):  # one Courant number per velocity column
        x = (-V + (j + 0.5) * 2 * V / nu[ax]) * dt / (A_HALF ** 2 * dx)
        col = f.select(3 + ax, j).movedim(ax, 0)
        shift = torch.tensor(abs(x), dtype=torch.float64, device=DEV)
        line = _advect(col if x >= 0 else col.flip(0), shift, True)
        line = line.roll(int(abs(x)), 0)
        col.copy_(line if x >= 0 else line.flip(0))


def _gradient(phi, d):
    n = phi.shape[d]
    r = lambda k: phi.roll(-k, d)  # noqa: E731
    return (8 * (r(1) - r(-1)) - (r(2) - r(-2))) * (n / (12 * BOX))


def _velocity_cells(f, ax, nu):
    """D_u of axis ax for cells f [m, nux, nuy, nuz] with Courant numbers nu [m]."""
    line = f.movedim(1 + ax, 0)
    neg = (nu < 0)[None, :, None, None]
    line = torch.where(neg, line.flip(0), line)
    out = _advect(line, nu.abs()[:, None, None], False)
    return torch.where(neg, out.flip(0), out).movedim(0, 1 + ax)


def _kick(f, phi, c, dt):
    """D_uz D_uy D_ux (dt) of Eq. (4) in place (FP64)."""
    n, nu = _sizes(c)
    cells = f.view((-1,) + nu)
    for ax in range(3):
        cour = (-_gradient(phi, ax) * dt * nu[ax] / (2 * c["V"])).reshape(-1)
        for i, j in _chunks(cells.shape[0], math.prod(nu)):
            cells[i:j] = _velocity_cells(cells[i:j], ax, cour[i:j])


def _rho(f, c):
    n, nu = _sizes(c)
    return f.view(n + (-1,)).sum(-1) * math.prod(2 * c["V"] / m for m in nu)


def _drift(f, c, dt):
    for ax in (2, 1, 0):
        _position(f, ax, c, dt)


def _exact_grad(c, s):
    """The run with every sweep's Jacobian taken by torch autograd, one sweep at a time."""
    n, nu = _sizes(c)
    dt, phi = s["dt"], s["phi"].double()
    ops = []
    for _ in range(c["steps"]):
        ops += [("u", 0), ("u", 1), ("u", 2), ("x", 2), ("x", 1), ("x", 0), ("u", 0), ("u", 1), ("u", 2)]
    f, kept = _initial(s["delta"], s["F"]).double(), []
    for op, ax in ops:
        kept.append(f)
        f = f.clone()
        if op == "x":
            _position(f, ax, c, dt)
        else:
            cour = (-_gradient(phi, ax) * (0.5 * dt) * nu[ax] / (2 * c["V"])).reshape(-1)
            cells = f.view((-1,) + nu)
            for i, j in _chunks(cells.shape[0], math.prod(nu)):
                cells[i:j] = _velocity_cells(cells[i:j], ax, cour[i:j])
    rho = _rho(f, c).requires_grad_(True)
    kx, ky, kz = _modes(n)
    k = torch.sqrt(kx * kx + ky * ky + kz * kz)
    loss = (torch.fft.fftn(rho).abs() ** 2 * ((k > 0) & (k < 8)).double()).sum()
    g, = torch.autograd.grad(loss, rho)
    lam = (g * math.prod(2 * c["V"] / m for m in nu))[..., None, None, None].expand(f.shape).clone()
    phi_g = phi.clone().requires_grad_(True)
    dphi = torch.zeros_like(phi)
    for op, ax in reversed(ops):
        x = kept.pop()
        if op == "x":
            for j in range(nu[ax]):
                cr = (-c["V"] + (j + 0.5) * 2 * c["V"] / nu[ax]) * dt * n[ax] / (A_HALF ** 2 * BOX)
                col = x.select(3 + ax, j).movedim(ax, 0)
                out = lam.select(3 + ax, j).movedim(ax, 0)
                flip = (lambda t: t) if cr >= 0 else (lambda t: t.flip(0))
                line = flip(col).clone().requires_grad_(True)
                new = _advect(line, torch.tensor(abs(cr), dtype=torch.float64, device=DEV), True)
                back, = torch.autograd.grad(new, line, flip(out))
                out.copy_(flip(back))
        else:
            cour = (-_gradient(phi_g, ax) * (0.5 * dt) * nu[ax] / (2 * c["V"])).reshape(-1)
            dcour = torch.zeros_like(cour)
            cells, lc = x.view((-1,) + nu), lam.view((-1,) + nu)
            for i, j in _chunks(cells.shape[0], math.prod(nu)):
                part = cells[i:j].clone().requires_grad_(True)
                cr = cour[i:j].detach().clone().requires_grad_(True)
                back = torch.autograd.grad(_velocity_cells(part, ax, cr), (part, cr), lc[i:j])
                lc[i:j] = back[0]
                dcour[i:j] = back[1]
            g, = torch.autograd.grad(cour, phi_g, dcour)
            dphi += g
    ddelta = torch.stack([(lam[i] * s["F"].double()).sum((-3, -2, -1)) for i in range(n[0])])
    return {"rho": rho.detach(), "ddelta": ddelta, "dphi": dphi}


def exact(case, seed):
    c = dict(case)
    n, nu = _sizes(c)
    cells = math.prod(n) * math.prod(nu)
    if cells > 2e9:
        return None
    s = _inputs(c, seed)
    kind = c["kind"]
    if kind == "codec":
        f = s["f"]
        scale = f.amax(-1)
        return {"codes": None, "scale": scale.double(), "f": f.double()}
    if kind == "moments":
        f = s["f"].view(n + nu)
        u = [_centres(m, -c["V"], c["V"]) for m in nu]
        S = torch.zeros((10,) + n, dtype=torch.float64, device=DEV)
        w = [torch.ones(nu, dtype=torch.float64, device=DEV)]
        U = [u[0][:, None, None].expand(nu), u[1][None, :, None].expand(nu), u[2].expand(nu)]
        w += U + [U[a] * U[b] for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
        W = torch.stack([x.reshape(-1) for x in w], 1)
        for ix in range(n[0]):
            S[:, ix] = (f[ix].reshape(n[1] * n[2], -1).double() @ W).T.reshape(10, n[1], n[2])
        um = S[1:4] / S[0]
        pair = torch.stack([um[a] * um[b] for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])
        return {"rho": S[0] * math.prod(2 * c["V"] / m for m in nu), "umean": um, "sigma2": S[4:] / S[0] - pair}
    if kind == "grad":
        out = _exact_grad(c, s)
        if c["dtype"] == "f32":
            # the gradient is discontinuous where a limiter changes branch: two FP32 runs that
            # round differently are 4e-4 .. 2e-3 from it by chance, with few cells carrying it
            # all, so the distance says nothing of either (FP64 draws compare the gradient)
            out["ddelta"] = out["dphi"] = None
        return out
    if c["dtype"] in ("bf16", "f16"):
        # the run starts from the codes: their values, rounded once to nearest
        f32 = s.pop("f")
        scale = f32.amax(-1, keepdim=True)
        if c["dtype"] == "bf16":
            scale = scale.clamp(min=2.0 ** -64)
        f = (f32 / scale).to(DTYPES[c["dtype"]]).double() * scale.double()
        del f32
    else:
        f = s.pop("f").double()
    if kind == "drift":
        _drift(f, c, s["dt"])
        return {"f": f}
    dt, phi = s["dt"], s["phi"].double()
    _kick(f, phi, c, 0.5 * dt)
    _drift(f, c, dt)
    rho = _rho(f, c)
    if c["sc"]:
        phi = _poisson(rho + s["bg"], A_FULL)
        phi32 = phi.float().double()  # the solver keeps its potential in FP32
    else:
        phi32 = phi
    _kick(f, phi32, c, 0.5 * dt)
    coded = c["dtype"] in ("bf16", "f16")
    out = {"f": None if coded else f, "rho": rho}
    if coded:
        out["scale"] = f.amax(-1)
    if c["sc"]:
        out["phi"] = phi
    return out
