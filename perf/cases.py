"""The work that programs have this library do, as measurable cases.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes what a program holds before the call (seeded fields on the
GPU, the plan or the simulation), ``run`` is one pass through the public entry
points, ``work`` what the pass cannot do without, and ``exact`` the same
outputs in 64 bits from torch and numpy alone.

Kinds of case:
  deriv     fc_deriv_z on a batch of physical fields (d/dz and d2/dz2)
  steps     a simulation run: set_fields, some RK3 steps, get_fields
  rhs       ns_rhs of physical fields
  project   fc_poisson_project of a stage's pressureless velocity
  ensemble  independent channel instances stepped together (Batch)
  noise     fc_noise, the App. A initial perturbation
"""
from __future__ import annotations

import decimal
import functools
import math

import numpy as np
import torch

from paper_2002_01392_gb300 import api

D, C = 5, 25                       # continuation order and points of every case
XY = (32, 64, 96, 128, 192, 256, 512)   # x / y lengths the drawn simulations take
ENSEMBLE = ((64, 64, 65), (96, 96, 97), (128, 128, 129), (192, 192, 129))


def listed():
    return [
        # the smallest channel grid's derivative: a call is a launch and its latency
        dict(name="deriv_32x32x33", kind="deriv", Nx=32, Ny=32, Nz=33, batch=3, prec="f32"),
        # three velocity components on a large grid: the benchmark's derivative
        dict(name="deriv_512x512x513", kind="deriv", Nx=512, Ny=512, Nz=513, batch=3, prec="f32"),
        # odd line counts (no two z-lines share an aligned vector), a convection run's Nz
        dict(name="deriv_255x129x103_odd", kind="deriv", Nx=255, Ny=129, Nz=103, batch=4, prec="f32"),
        # the paper's precision
        dict(name="deriv_256x256x513_f64", kind="deriv", Nx=256, Ny=256, Nz=513, batch=3, prec="f64"),
        # a small served channel simulation: latency of many short kernels
        dict(name="steps_64x64x65", kind="steps", Nx=64, Ny=64, Nz=65, nfields=3, prec="f32", steps=4),
        # a channel run in the paper's precision
        dict(name="steps_128x128x129_f64", kind="steps", Nx=128, Ny=128, Nz=129, nfields=3, prec="f64", steps=2),
        # the largest served grid, Boussinesq
        dict(name="steps_256x256x257", kind="steps", Nx=256, Ny=256, Nz=257, nfields=4, prec="f32", steps=4),
        # the large convection grid (half of it in y, so that three runs fit the card)
        dict(name="steps_1024x512x513", kind="steps", Nx=1024, Ny=512, Nz=513, nfields=4, prec="f32", steps=2),
        # the right-hand side alone, as a user's own time stepper calls it
        dict(name="rhs_192x192x129", kind="rhs", Nx=192, Ny=192, Nz=129, nfields=4, prec="f32"),
        # the pressure projection alone: half of the served requests
        dict(name="project_256x256x257", kind="project", Nx=256, Ny=256, Nz=257, nfields=3, prec="f32"),
        # an ensemble of uneven channel instances, one graph launch per step
        dict(name="ensemble_16", kind="ensemble", members=16, steps=2, prec="f32", pick=0),
        # the initial perturbation of a run
        dict(name="noise_512x512x257", kind="noise", Nx=512, Ny=512, Nz=257, prec="f32"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("deriv", "deriv", "deriv", "steps", "steps", "rhs", "project", "ensemble", "noise"))
    prec = "f64" if rng.random() < 0.25 else "f32"
    if kind == "deriv":
        batch = rng.randint(1, 4)
        Nz = rng.choice((_logint(rng, 33, 750), rng.choice((39, 103, 231, 479, 487, 513, 999))))
        most = (2.5e8 if prec == "f32" else 2.5e7) / (Nz * batch)
        Nx = _logint(rng, 17, 512)
        Ny = max(1, min(_logint(rng, 17, 512), int(most / Nx)))
        return dict(kind=kind, Nx=Nx, Ny=Ny, Nz=Nz, batch=batch, prec=prec)
    if kind == "ensemble":
        return dict(kind=kind, members=rng.randint(2, 24), steps=rng.randint(1, 3), prec="f32",
                    pick=rng.randint(1, 1000))
    if kind == "noise":
        return dict(kind=kind, Nx=_logint(rng, 33, 512), Ny=_logint(rng, 33, 512), Nz=_logint(rng, 33, 300), prec=prec)
    most = 3.4e7 if prec == "f32" else 2.2e6
    while True:
        Nx, Ny, Nz = rng.choice(XY), rng.choice(XY), _logint(rng, 33, 263)
        if rng.random() < 0.2:
            Nx = 1024 if prec == "f32" else 512
        if Nx * Ny * Nz <= most and Nz + C <= 288:
            break
    nf = 3 if kind == "project" else rng.choice((3, 4))
    case = dict(kind=kind, Nx=Nx, Ny=Ny, Nz=Nz, nfields=nf, prec=prec)
    if kind == "steps":
        case["steps"] = rng.randint(1, 4)
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _dtype(case):
    return torch.float64 if case["prec"] == "f64" else torch.float32


def _modes(g, Nx, Ny, slope):
    """A real [Ny][Nx] field of random-phase modes, amplitudes |k|^slope up to the 2/3 cutoff, and its x, y
    derivatives and horizontal Laplacian; the largest value is 1."""
    kx = torch.fft.rfftfreq(Nx, 1.0 / Nx, device="cuda", dtype=torch.float64)[None, :]
    ky = torch.fft.fftfreq(Ny, 1.0 / Ny, device="cuda", dtype=torch.float64)[:, None]
    k = torch.sqrt(kx * kx + ky * ky)
    keep = (k > 0) & (3 * kx.abs() <= Nx) & (3 * ky.abs() <= Ny)
    amp = torch.where(keep, k.clamp(min=1.0) ** slope, torch.zeros_like(k))
    ph = 2 * math.pi * torch.rand(k.shape, generator=g, device="cuda", dtype=torch.float64)
    s = torch.polar(amp, ph)
    back = lambda q: torch.fft.irfft2(q, s=(Ny, Nx)) * (Nx * Ny)  # noqa: E731
    f = back(s)
    c = 1.0 / f.abs().max()
    return [c * back(q) for q in (s, 1j * kx * s, 1j * ky * s, -k * k * s)]


def _deriv_field(case, seed):
    """A turbulent field: eight products of a Kolmogorov-spectrum horizontal field and a vertical profile, which
    is smooth in the sublayer at the walls (six points) and carries an inertial-range spectrum up to the 2/3 cutoff
    outside it."""
    g = _gen(seed)
    Nx, Ny, Nz = case["Nx"], case["Ny"], case["Nz"]
    z = torch.arange(Nz, device="cuda", dtype=torch.float64) / (Nz - 1)
    K = max(1, 2 * (Nz - 1) // 3)
    k = torch.arange(1, K + 1, device="cuda", dtype=torch.float64)
    n = torch.arange(1 + min(16, Nz // 10), device="cuda", dtype=torch.float64)
    cheb = torch.cos(n[:, None] * torch.arccos((2 * z - 1).clamp(-1, 1))[None, :])
    i = torch.arange(Nz, device="cuda", dtype=torch.float64)
    i = torch.minimum(i, Nz - 1 - i)
    damp = torch.sin(0.5 * math.pi * ((i - 5) / 10).clamp(0, 1)) ** 2
    out = torch.empty((case["batch"], Nz, Ny, Nx), device="cuda", dtype=_dtype(case))
    for b in range(case["batch"]):
        X = torch.stack([_modes(g, Nx, Ny, -4.0 / 3.0)[0] for _ in range(8)])
        coef = torch.randn((8, n.numel()), generator=g, device="cuda", dtype=torch.float64) * 2.0 ** (-n / 2)
        ph = 2 * math.pi * torch.rand((8, K, 1), generator=g, device="cuda", dtype=torch.float64)
        rough = (k[None, :, None] ** (-5.0 / 6.0) * torch.cos(math.pi * k[None, :, None] * z[None, None, :] + ph)).sum(1)
        Z = coef @ cheb + damp * rough
        torch.matmul(Z.T.to(out.dtype), X.reshape(8, -1).to(out.dtype), out=out[b].view(Nz, Ny * Nx))
    return out


def _flow(case, seed, nf):
    """A solenoidal no-slip velocity curl(psi z) + curl curl(chi z) of Kolmogorov horizontal spectra: on the
    laminar profile (channel), or with a temperature that vanishes at the walls (Boussinesq).  For the projection, the
    pressureless velocity of a stage: a part that is neither solenoidal nor impermeable is added."""
    g = _gen(seed)
    Nx, Ny, Nz = case["Nx"], case["Ny"], case["Nz"]
    z = torch.arange(Nz, device="cuda", dtype=torch.float64) / (Nz - 1)
    a = torch.rand(3, generator=g, device="cuda", dtype=torch.float64) * 2 - 1
    p = z * (1 - z) * (1 + a[0] * z + a[1] * z * z)
    w = z * (1 - z)
    q = w * w * (1 + a[2] * z)
    dq = 2 * w * (1 - 2 * z) * (1 + a[2] * z) + w * w * a[2]
    _, px, py, _ = _modes(g, Nx, Ny, -7.0 / 3.0)
    _, cx, cy, cl = _modes(g, Nx, Ny, -10.0 / 3.0)
    out = torch.empty((nf, Nz, Ny, Nx), device="cuda", dtype=_dtype(case))
    t = out.dtype
    outer = lambda prof, f: prof.to(t)[:, None, None] * f.to(t)[None]  # noqa: E731
    out[0] = outer(p, py)
    out[0] += outer(dq, cx)
    out[1] = outer(-p, px)
    out[1] += outer(dq, cy)
    out[2] = outer(-q, cl)
    out[:3] *= 0.3 / max(float(out[i].abs().max()) for i in range(3))
    if nf == 4:
        out[3] = outer(0.3 * torch.sin(math.pi * z), _modes(g, Nx, Ny, -4.0 / 3.0)[0])
    else:
        out[0] += (5.0 * z * (1 - z)).to(t)[:, None, None]
    if case.get("kind") == "project":
        X = _modes(g, Nx, Ny, -4.0 / 3.0)[0]
        for i in range(3):
            out[i] += outer(0.1 * torch.cos(math.pi * (i + 1) * z), X.roll(5 * i, 1))
    return out


def _nu(Nz):
    """Ra = 1e7 (Pr = 1) at Nz = 129; finer grids are there for larger Ra: Nz ~ Ra^0.3."""
    return 3.162e-4 * (129 / Nz) ** (5.0 / 3.0)


def _physics(nf, Nz):
    nu = _nu(Nz)
    if nf == 4:
        return dict(nfields=4, nu=nu, kappa=nu, gamma=1.0)
    return dict(nfields=3, nu=nu, forcing_x=10 * nu)


def _dt(Nz):
    return min(1e-3, 0.5 / (3e-3 * (math.pi * (Nz - 1)) ** 2))   # inside the explicit viscous limit


def _members(case):
    r = np.random.Generator(np.random.PCG64(2002 + case["pick"]))
    return [dict(zip(("Nx", "Ny", "Nz"), ENSEMBLE[int(r.integers(0, 4))]), prec=case["prec"],
                 nu=float(np.exp(r.uniform(math.log(1e-3), math.log(3e-3))))) for _ in range(case["members"])]


def _sim(c, phys):
    return api.Sim(api.ns_params(Nx=c["Nx"], Ny=c["Ny"], Nz=c["Nz"], d=D, C=C, prec=c["prec"], **phys))


def _draws(par, seed):
    return np.random.Generator(np.random.PCG64(seed)).uniform(size=2 * api.noise_modes(par))


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind)
    if kind == "deriv":
        s["plan"] = api.Plan(D, C, case["Nz"])
        s["f"] = _deriv_field(case, seed)
        s["df"], s["d2f"] = torch.empty_like(s["f"]), torch.empty_like(s["f"])
    elif kind == "noise":
        s["par"] = api.noise_params(amplitude=1e-3)
        s["draws"] = _draws(s["par"], seed)
        s["out"] = torch.empty((3, case["Nz"], case["Ny"], case["Nx"]), device="cuda", dtype=_dtype(case))
    elif kind == "ensemble":
        ms = _members(case)
        s["phys"] = [_flow(m, seed + 1000 * i, 3) for i, m in enumerate(ms)]
        s["sims"] = [_sim(m, dict(_physics(3, m["Nz"]), nu=m["nu"])) for m in ms]
        s["batch"] = api.Batch(s["sims"])
        s["dt"] = [_dt(m["Nz"]) for m in ms]
        s["steps"] = case["steps"]
        s["out"] = [torch.empty_like(p) for p in s["phys"]]
    else:
        nf = case["nfields"]
        s["phys"] = _flow(case, seed, nf)
        s["sim"] = _sim(case, _physics(nf, case["Nz"]))
        s["sim"].tune(1)
        s["dt"] = _dt(case["Nz"])
        s["steps"] = case.get("steps", 1)
        s["out"] = torch.empty_like(s["phys"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "deriv":
        return api.fc_deriv_z(s["plan"], s["f"], s["df"], s["d2f"])
    if kind == "noise":
        return api.fc_noise(s["par"], s["draws"], s["out"])
    if kind == "rhs":
        return s["sim"].rhs(s["phys"], s["out"])
    if kind == "project":
        return s["sim"].project(s["phys"], s["dt"], s["out"])
    if kind == "ensemble":
        for sim, p in zip(s["sims"], s["phys"]):
            sim.set_fields(p)
        for _ in range(s["steps"]):
            s["batch"].step(s["dt"])
        for sim, o in zip(s["sims"], s["out"]):
            sim.get_fields(o)
        return s["out"]
    s["sim"].set_fields(s["phys"])
    for _ in range(s["steps"]):
        s["sim"].step(s["dt"])
    return s["sim"].get_fields(s["out"])


def work(case):
    """Bytes: inputs read once, outputs written once, and for every Runge-Kutta stage the fields read twice (step
    and stage values) and written once.  Flops: 5/2 N log2 N per real transform, of z-lines for the derivatives,
    of all three directions elsewhere."""
    kind = case["kind"]
    if kind == "ensemble":
        parts = [work(dict(m, kind="steps", nfields=3, steps=case["steps"])) for m in _members(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    es = 8 if case["prec"] == "f64" else 4
    pts = case["Nx"] * case["Ny"] * case["Nz"]
    lg = math.log2
    if kind == "deriv":
        Np = case["Nz"] + C
        lines = case["Nx"] * case["Ny"] * case["batch"]
        return {"bytes": 3.0 * es * pts * case["batch"], "flops": lines * (3 * 2.5 * Np * lg(Np) + 4.0 * D * C)}
    if kind == "noise":
        return {"bytes": 3.0 * es * pts, "flops": 3.0 * pts * 4}
    nf = case["nfields"]
    fft = 2.5 * pts * lg(pts)      # one field through all three directions
    if kind == "project":
        return {"bytes": 6.0 * es * pts, "flops": 6 * fft}
    stage = nf * 5 * fft           # v, three gradients, the nonlinear term
    if kind == "rhs":
        return {"bytes": 2.0 * nf * es * pts, "flops": nf * 2 * fft + stage}
    n = 3 * case["steps"]
    return {"bytes": (2.0 + 3.0 * n) * nf * es * pts, "flops": nf * 2 * fft + n * (stage + nf * fft)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from torch and numpy
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _continuation_matrix(d, c):
    """M_r (c x d): least-squares Fourier continuation of the d Lagrange polynomials of the points 0..d-1 (period
    2 (d + c), bandwidth 2 (d + c) / 3, 20 samples per grid interval, zero on the mirrored points), at 80 digits."""
    with decimal.localcontext() as ctx:
        ctx.prec = 80
        Dc = decimal.Decimal

        def atan_inv(n):
            x = Dc(1) / n
            s, t, k = x, x, 1
            while abs(t) > Dc(10) ** -82:
                t = -t / (n * n)
                k += 2
                s += t / k
            return s

        pi = 4 * (4 * atan_inv(5) - atan_inv(239))   # Machin's formula

        def cos_sin(x):
            x = x % (2 * pi)
            co, si, t, k = Dc(0), Dc(0), Dc(1), 0
            while abs(t) > Dc(10) ** -82 or k < 20:
                if k % 2 == 0:
                    co += t if k % 4 == 0 else -t
                else:
                    si += t if k % 4 == 1 else -t
                k += 1
                t = t * x / k
            return co, si

        M, n_os, P = 2 * (d + c) // 3, 20, 2 * (d + c)
        # every abscissa is an integer over n_os: the cosines of all multiples of 2 pi / (P n_os)
        tab = [cos_sin(2 * pi * j / (P * n_os)) for j in range(P * n_os)]

        def row(j):   # abscissa j / n_os
            r = [Dc(1)]
            for m in range(1, M + 1):
                r += tab[(m * j) % (P * n_os)]
            return r

        right = list(range((d - 1) * n_os + 1))
        left = [(d + c) * n_os + j for j in right]
        cols = [list(v) for v in zip(*[row(j) for j in right + left])]
        ncol = len(cols)
        R = [[Dc(0)] * ncol for _ in range(ncol)]
        dot = lambda u, v: sum((x * y for x, y in zip(u, v)), Dc(0))  # noqa: E731
        for i in range(ncol):   # modified Gram-Schmidt: cols becomes Q
            R[i][i] = dot(cols[i], cols[i]).sqrt()
            cols[i] = [x / R[i][i] for x in cols[i]]
            for j in range(i + 1, ncol):
                R[i][j] = dot(cols[i], cols[j])
                cols[j] = [y - R[i][j] * x for x, y in zip(cols[i], cols[j])]
        out = np.empty((c, d))
        rows = [row((d + j) * n_os) for j in range(c)]
        for i in range(d):
            b = []
            for j in right:
                v = Dc(1)
                for q in range(d):
                    if q != i:
                        v = v * (Dc(j) / n_os - q) / (i - q)
                b.append(v)
            b += [Dc(0)] * len(left)
            x = [Dc(0)] * ncol
            for k in range(ncol):
                x[k] = dot(cols[k], b)
                b = [u - x[k] * v for u, v in zip(b, cols[k])]
            for k in range(ncol - 1, -1, -1):
                x[k] = (x[k] - dot(R[k][k + 1:], x[k + 1:])) / R[k][k]
            for j in range(c):
                out[j, i] = float(dot(rows[j], x))
    return out


class _Ref:
    """The method in float64 on the GPU: fields in (x, y, z), transforms by torch.fft, states continued in z."""

    def __init__(self, Nx, Ny, Nz, nu=0.0, kappa=0.0, gamma=0.0, forcing_x=0.0, nfields=3):
        f64 = dict(device="cuda", dtype=torch.float64)
        self.Nx, self.Ny, self.Nz, self.Np = Nx, Ny, Nz, Nz + C
        self.dif, self.gamma, self.F, self.nf = [nu, nu, nu, kappa], gamma, forcing_x, nfields
        self.Mr = torch.tensor(_continuation_matrix(D, C), **f64)
        self.Ml = self.Mr.flip(0, 1)
        kx = torch.arange(Nx // 2 + 1, **f64)
        ky = torch.fft.fftfreq(Ny, 1.0 / Ny, **f64)
        nz = torch.fft.fftfreq(self.Np, 1.0 / self.Np, **f64)
        kz = 2 * math.pi * nz * (Nz - 1) / self.Np

        def odd(k, n):
            k = k.clone()
            if n % 2 == 0:
                k[n // 2] = 0
            return k

        self.kx, self.ky, self.kz = kx[None, None, :], ky[None, :, None], kz[:, None, None]
        self.ox, self.oy, self.oz = (odd(kx, Nx)[None, None, :], odd(ky, Ny)[None, :, None],
                                     odd(kz, self.Np)[:, None, None])
        fz = torch.exp(-16 * math.log(10.0) * (nz.abs() / (self.Np / 2)) ** 100)[:, None, None]
        self.filt = fz * ((3 * ky.abs() <= Ny).double()[None, :, None] * (3 * kx <= Nx).double()[None, None, :])
        self.z = (torch.arange(Nz, **f64) / (Nz - 1))[:, None, None]

    def extend(self, m):
        """[Nz, ...] -> [N', ...] along the first axis."""
        a, b = m[:D].reshape(D, -1), m[-D:].reshape(D, -1)
        e = self.Mr.to(m.dtype) @ b + self.Ml.to(m.dtype) @ a
        return torch.cat([m, e.reshape((C,) + m.shape[1:])])

    def fwd(self, phys):
        return torch.fft.fft(self.extend(torch.fft.fft(torch.fft.rfft(phys, dim=2), dim=1)), dim=0)

    def inz(self, s):
        return torch.fft.ifft(s, dim=0)[:self.Nz]

    def phys(self, m):
        return torch.fft.irfft(torch.fft.ifft(m, dim=1), n=self.Nx, dim=2)

    def nonlinear(self, st):
        m = [self.inz(s) for s in st]
        v = [self.phys(q) for q in m[:3]]
        out = []
        for c in range(self.nf):
            n = -v[0] * self.phys(1j * self.ox * m[c])
            n -= v[1] * self.phys(1j * self.oy * m[c])
            n -= v[2] * self.phys(self.inz(1j * self.oz * st[c]))
            if c == 0:
                n += self.F
            if self.nf == 4 and c == 2:
                n += self.gamma * self.phys(m[3])
            if c == 3:
                n += self.gamma * v[2]
            out.append(self.fwd(n) * self.filt)
        return out

    def lap(self, c):
        return self.dif[c] * (self.kx ** 2 + self.ky ** 2 + self.kz ** 2)

    def stage(self, m, dtj, gp):
        """Injection at the walls, continuation and projection of the mixed values m; the new state and planes."""
        for w, s in ((0, 0), (1, self.Nz - 1)):
            m[0][s], m[1][s] = dtj * gp[w, 0], dtj * gp[w, 1]
            if len(m) == 4:
                m[3][s] = 0
        st = [torch.fft.fft(self.extend(q), dim=0) for q in m]
        kk = self.ox ** 2 + self.oy ** 2 + self.oz ** 2
        s = (self.ox * st[0] + self.oy * st[1] + self.oz * st[2]) / torch.where(kk > 0, kk, torch.ones_like(kk))
        s = torch.where(kk > 0, s, torch.zeros_like(s))
        del kk
        wz = self.inz(st[2] - self.oz * s)
        b, t = wz[0], wz[-1]
        g = torch.sqrt(self.ox[0] ** 2 + self.oy[0] ** 2)
        E = torch.exp(-g)
        flat = g == 0
        den = torch.where(flat, torch.ones_like(g), g * (1 - E * E))
        zero = torch.zeros_like(b)
        A = torch.where(flat, zero, (t - b * E) / den)
        B = torch.where(flat, zero, -(b - t * E) / den)
        Dm = torch.where(flat, 0.5 * (b + t), zero)
        e1, e2 = torch.exp(g * (self.z - 1)), torch.exp(-g * self.z)
        Phi = A * e1 + B * e2
        grads = [1j * self.ox * Phi, 1j * self.oy * Phi, g * (A * e1 - B * e2) + Dm]
        new = torch.empty_like(gp)
        gI = self.inz(s)
        for w, zi in ((0, 0), (1, self.Nz - 1)):
            new[w, 0] = (self.ox[0] * gI[zi] + grads[0][zi]) / dtj
            new[w, 1] = (self.oy[0] * gI[zi] + grads[1][zi]) / dtj
        del gI, Phi, e1, e2, wz
        for c, k in enumerate((self.ox, self.oy, self.oz)):
            st[c] -= k * s
            st[c] -= torch.fft.fft(self.extend(grads[c]), dim=0)
        return st, new

    def planes(self):
        return torch.zeros((2, 2, self.Ny, self.Nx // 2 + 1), device="cuda", dtype=torch.complex128)

    def steps(self, phys, dt, n):
        st, gp = [self.fwd(p.double()) for p in phys], self.planes()
        for _ in range(n):
            v0 = vj = st
            for j in range(1, 4):
                dtj = dt / (4 - j)
                N = self.nonlinear(vj)
                m = []
                for c in range(self.nf):
                    m.append(self.inz(v0[c] + dtj * (N[c] - self.lap(c) * vj[c])))
                    N[c] = None
                vj, gp = self.stage(m, dtj, gp)
            st = vj
        return torch.stack([self.phys(self.inz(s)) for s in st])

    def rhs(self, phys):
        st = [self.fwd(p.double()) for p in phys]
        N = self.nonlinear(st)
        return torch.stack([self.phys(self.inz(N[c] - self.lap(c) * st[c])) for c in range(self.nf)])

    def project(self, phys, dtj):
        m = [torch.fft.fft(torch.fft.rfft(p.double(), dim=2), dim=1) for p in phys]
        st, _ = self.stage(m, dtj, self.planes())
        return torch.stack([self.phys(self.inz(s)) for s in st])


def _exact_deriv(case, seed):
    f = _deriv_field(case, seed)
    Nz, Np = case["Nz"], case["Nz"] + C
    r = _Ref(2, 2, Nz)
    ident = torch.eye(Nz, device="cuda", dtype=torch.float64)
    spec = torch.fft.fft(r.extend(ident), dim=0)
    out = []
    for fac in (1j * r.oz[:, 0], -r.kz[:, 0] ** 2):
        op = torch.fft.ifft(spec * fac, dim=0)[:Nz].real.contiguous()
        out.append(torch.stack([(op @ b.reshape(Nz, -1).double()).reshape(b.shape) for b in f]))
    return out


def _exact_noise(case, seed):
    par = api.noise_params(amplitude=1e-3)
    u = _draws(par, seed)
    Nx, Ny, Nz = case["Nx"], case["Ny"], case["Nz"]
    zp = np.arange(Nz) / (Nz - 1) - 0.5

    def root(m):   # tanh t + tan t = 0 (m odd) or tanh t - tan t = 0 (m even) on the m-th bracket, lambda = 2 t
        j = (m + 1) // 2 if m % 2 else m // 2
        lo, hi = (j * math.pi - math.pi / 2 + 1e-9, j * math.pi) if m % 2 else (j * math.pi, j * math.pi + math.pi / 2 - 1e-9)
        f = lambda t: math.tanh(t) + (math.tan(t) if m % 2 else -math.tan(t))  # noqa: E731
        up = f(hi) > 0
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            if (f(mid) > 0) == up:
                hi = mid
            else:
                lo = mid
        return lo + hi

    lam = {m: root(m) for m in range(2, 6)}
    Q = {}
    i = 0
    for n in range(-6, 7):
        for l in range(0, 7):
            if (l == 0 and n <= 0) or not 4 <= n * n + l * l <= 25:
                continue
            pr = np.zeros((3, Nz), dtype=np.complex128)
            for m in range(2, 6):
                L = lam[m]
                k = math.sqrt(n * n + l * l + L * L)
                a = k ** -4.0 * np.exp(2j * math.pi * u[i])
                b = k ** -3.0 * np.exp(2j * math.pi * u[i + 1])
                i += 2
                if m % 2:
                    g = np.cosh(L * zp) / math.cosh(L / 2) - np.cos(L * zp) / math.cos(L / 2)
                    dg = L * (np.sinh(L * zp) / math.cosh(L / 2) + np.sin(L * zp) / math.cos(L / 2))
                else:
                    g = np.sinh(L * zp) / math.sinh(L / 2) - np.sin(L * zp) / math.sin(L / 2)
                    dg = L * (np.cosh(L * zp) / math.sinh(L / 2) - np.cos(L * zp) / math.sin(L / 2))
                s = np.sin(m * math.pi * (zp + 0.5))
                pr[0] += 1j * n * a * dg + 1j * l * b * s
                pr[1] += 1j * l * a * dg - 1j * n * b * s
                pr[2] += (n * n + l * l) * a * g
            Q[(n, l)] = pr
    ns, ls = range(-5, 6), range(0, 6)
    A = np.zeros((3, Nz, len(ls), len(ns)), dtype=np.complex128)
    for (n, l), pr in Q.items():
        A[:, :, l, n + 5] = pr
    A = torch.tensor(A, device="cuda")
    ang = lambda ks, N: torch.tensor([[(k * j) % N for j in range(N)] for k in ks], device="cuda", dtype=torch.float64) * (2 * math.pi / N)  # noqa: E731
    ex, ey = ang(ns, Nx), ang(ls, Ny)
    R = torch.einsum("czln,ly->czyn", A, torch.polar(torch.ones_like(ey), ey))
    q = torch.matmul(R.real, torch.cos(ex)) - torch.matmul(R.imag, torch.sin(ex))
    return q * (1e-3 / q.abs().max())


def exact(case, seed):
    kind = case["kind"]
    if kind == "deriv":
        return _exact_deriv(case, seed)
    if kind == "noise":
        return _exact_noise(case, seed)
    if kind == "ensemble":
        out = []
        for i, m in enumerate(_members(case)):
            r = _Ref(m["Nx"], m["Ny"], m["Nz"], **dict(_physics(3, m["Nz"]), nu=m["nu"]))
            out.append(r.steps(_flow(m, seed + 1000 * i, 3), _dt(m["Nz"]), case["steps"]))
        return out
    nf = case["nfields"]
    r = _Ref(case["Nx"], case["Ny"], case["Nz"], **_physics(nf, case["Nz"]))
    phys = _flow(case, seed, nf)
    if kind == "rhs":
        return r.rhs(phys)
    if kind == "project":
        return r.project(phys, _dt(case["Nz"]))
    return r.steps(phys, _dt(case["Nz"]), case["steps"])
