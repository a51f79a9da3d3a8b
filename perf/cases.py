"""Measured workloads of the library: scattering runs, batched sweeps and gradients.

A scattering pass is what a user's loop does once per period: put a DFT window
over the next period (T = 3 lambda steps), step through it, project the near
fields to the far field, and look at the total energy (the steady-state check)
and the field maps.  The state it starts from is a run under way: ``prepare``
takes the steps the incident wave needs to reach the scatterer.  A batched pass
does the same for many uneven problems, an adjoint pass is one evaluation of
far-field intensities and their gradient with respect to the permittivity.

``exact`` runs the same problems in plain FP64 torch (total-field form of the
scheme, link-wise total-field/scattered-field source).
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2510_11042_gb300 import lbem
from paper_2510_11042_gb300.autograd import far_field_intensity

SIGMA_MAX = 0.3
RAMP_PERIODS = 3.0


def listed():
    scatter = dict(kind="scatter", mode="ez", storage="f32", streaming="two_buffers", source="line", nz=1)
    return [
        # the planar dielectric interface at 30 degrees incidence: the smallest
        # grid in use, closed-form oblique source, no far field
        dict(scatter, name="planar_200_ez_f32", source="oblique", nx=200, ny=200, width=10, wavelength=40),
        # a 2D scatterer on one of the paper's ragged grids, TE polarisation
        dict(scatter, name="cylinder_520_hz_f32", mode="hz", nx=520, ny=520, width=20, wavelength=40),
        # the 2D cylinder configuration, TM polarisation
        dict(scatter, name="cylinder_1024_ez_f32", nx=1024, ny=1024, width=20, wavelength=40),
        # the paper's 1000^2 grid in reduced-precision storage, TE polarisation
        dict(scatter, name="cylinder_1000_hz_f16", mode="hz", storage="f16", nx=1000, ny=1000, width=20,
             wavelength=40),
        # the paper's largest 2D grid (a cylinder of many wavelengths)
        dict(scatter, name="cylinder_4000_ez_f32", nx=4000, ny=4000, width=20, wavelength=40),
        # the small 3D sphere (the parity subproblem's size)
        dict(scatter, name="sphere_64_f32", mode="3d", nx=64, ny=64, nz=64, width=8, wavelength=16),
        # the paper's 300^3 sphere on one population buffer, BF16 storage
        dict(scatter, name="sphere_300_bf16_in_place", mode="3d", storage="bf16", streaming="in_place", nx=300,
             ny=300, nz=300, width=16, wavelength=30),
        # the 3D sphere configuration in its two main storage types
        dict(scatter, name="sphere_384_f32", mode="3d", nx=384, ny=384, nz=384, width=16, wavelength=30),
        dict(scatter, name="sphere_384_f16", mode="3d", storage="f16", nx=384, ny=384, nz=384, width=16,
             wavelength=30),
        # the batched sweep: 32 cylinders on uneven grids
        dict(kind="batch", name="batch_32_cylinders", storage="f32", count=32, lo=256, hi=1024, sizes=20251011),
        # the hexagon-sized gradient: 4000 steps, a checkpoint every 200
        dict(kind="adjoint", name="adjoint_512_ez", mode="ez", nx=512, ny=512, nz=1, width=20, wavelength=40,
             steps=4000, every=200, angles=3),
        # a 3D gradient
        dict(kind="adjoint", name="adjoint_96_3d", mode="3d", nx=96, ny=96, nz=96, width=8, wavelength=8, steps=384,
             every=48, angles=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(("2d", "2d", "2d", "2d", "3d", "3d", "3d", "batch", "adjoint", "adjoint"))
    if what == "batch":
        lo = _log(rng, 64, 256)
        return dict(kind="batch", storage=rng.choice(("f32", "f32", "f16")), count=rng.randint(4, 32), lo=lo,
                    hi=_log(rng, lo + 32, 1024), sizes=rng.randrange(1 << 30))
    if what == "adjoint":
        if rng.random() < 0.6:
            n = _log(rng, 128, 512)
            return dict(kind="adjoint", mode=rng.choice(("ez", "hz")), nx=n, ny=_log(rng, 128, 512), nz=1, width=12,
                        wavelength=rng.randint(10, 40), steps=_log(rng, 4 * n, 4000), every=rng.randint(50, 200),
                        angles=rng.randint(1, 8))
        n = _log(rng, 48, 96)
        return dict(kind="adjoint", mode="3d", nx=_log(rng, 48, 96), ny=_log(rng, 48, 96), nz=n, width=6, wavelength=8,
                    steps=rng.randint(3 * n + 24, 4 * n), every=rng.randint(20, 60), angles=3)
    case = dict(kind="scatter", storage=rng.choice(("f32", "f32", "f16", "bf16")), streaming="two_buffers",
                source="line")
    if what == "2d":
        case.update(mode=rng.choice(("ez", "hz")), nx=_log(rng, 200, 4000), ny=_log(rng, 200, 4000), nz=1,
                    width=rng.randint(10, 20), wavelength=rng.randint(20, 40))
        if case["nx"] * case["ny"] < 1 << 19 and rng.random() < 0.25:
            case["source"] = "oblique"
        return case
    case.update(mode="3d", nx=_log(rng, 64, 384), ny=_log(rng, 64, 384), nz=_log(rng, 64, 384),
                width=rng.randint(8, 16), wavelength=rng.randint(12, 30))
    if rng.random() < 0.2:
        case["streaming"] = "in_place"
    return case


# ------------------------------------------------------------- the problems
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _wave(case):
    """Line source: +x in 2D, +z in 3D, boxes 4 cells apart inside the layer.
    Oblique: the closed-form wave at 30 degrees on the one-sided region x >= 2 w."""
    n, w, lam, mode = (case["nx"], case["ny"], case["nz"]), case["width"], float(case["wavelength"]), case["mode"]
    if case.get("source") == "oblique":
        th = math.radians(30.0)
        pol = (0.0, 0.0, 1.0) if mode == "ez" else (-math.sin(th), math.cos(th), 0.0)
        return SimpleNamespace(direction=(math.cos(th), math.sin(th), 0.0), polarization=pol, wavelength=lam,
                               amplitude=1.0, ramp_periods=RAMP_PERIODS, tf_lo=(2 * w, w + 5, 0),
                               tf_hi=(10 ** 6, n[1] - 1 - w - 5, 0), ntff_lo=(0, 0, 0), ntff_hi=(0, 0, 0),
                               center=(0.0, 0.0, 0.0), source_index=-1, analytic=True,
                               origin=(2.0 * w, 0.0, 0.0))
    at = lambda side, gap: tuple(0 if m == 1 else (w + gap if side == 0 else m - 1 - w - gap) for m in n)  # noqa: E731
    d, p = {"ez": ((1.0, 0.0, 0.0), (0.0, 0.0, 1.0)), "hz": ((1.0, 0.0, 0.0), (0.0, 1.0, 0.0)),
            "3d": ((0.0, 0.0, 1.0), (1.0, 0.0, 0.0))}[mode]
    return SimpleNamespace(direction=d, polarization=p, wavelength=lam, amplitude=1.0, ramp_periods=RAMP_PERIODS,
                           ntff_lo=at(0, 4), ntff_hi=at(1, 4), tf_lo=at(0, 8), tf_hi=at(1, 8),
                           center=tuple((m - 1) / 2.0 for m in n), source_index=w + 2, analytic=False,
                           origin=(0.0, 0.0, 0.0))


def _eps(case, seed):
    """A dielectric half-space (oblique) or a round body near the centre, with
    the permittivity, the size and the place drawn from the seed."""
    rng = random.Random("%d %s" % (seed, sorted((k, v) for k, v in case.items() if k != "name")))
    n, w, dev = (case["nx"], case["ny"], case["nz"]), case["width"], _device()
    eps_in = rng.uniform(1.5, 4.0)
    if case.get("source") == "oblique":
        eps = torch.ones((1, n[1], n[0]), dtype=torch.float32, device=dev)
        eps[:, :, n[0] // 2 + rng.randint(-5, 5):] = eps_in
        return eps
    room = min(m for m in n if m > 1) / 2.0 - w - 12
    a = max(2.0, min(room - 3.0, rng.uniform(0.5, 1.0) * min(room, 1.2 * case["wavelength"])))
    x, y, z = (torch.arange(m, device=dev, dtype=torch.float32) - ((m - 1) / 2.0 + (rng.uniform(-2, 2) if m > 1 else 0))
               for m in n)
    r2 = (x * x)[None, None, :] + (y * y)[None, :, None] + (z * z)[:, None, None]
    eps = torch.where(r2 <= a * a, eps_in, 1.0).to(torch.float32)
    if case["kind"] == "adjoint":  # a design in progress: every cell of the body differs
        g = torch.Generator(device=dev).manual_seed(rng.randrange(1 << 40))
        u = torch.rand(eps.shape, generator=g, device=dev) * 0.1 - 0.05
        eps = torch.where(eps > 1.0, eps * (1.0 + u), eps)
    return eps.contiguous()


def _period(case):
    return 3 * case["wavelength"]


def _warm(case):
    """Steps before the measured period: whole periods, past the scattered wave's
    arrival at the near-field box (c = 1/3 cell a step)."""
    along = case["nz"] if case["mode"] == "3d" else case["nx"]
    T = _period(case)
    return -(-(3 * along + T) // T) * T


def _angles(mode):
    theta = np.radians(np.arange(181.0))
    if mode != "3d":
        return theta, None
    return np.tile(theta, 3), np.repeat(np.radians([0.0, 45.0, 90.0]), 181)


def _batch_cases(case):
    """The problems of a sweep: square grids in multiples of 32, each with a wavelength of its own."""
    rng = random.Random(case["sizes"])
    small = case["hi"] < 256
    return [dict(kind="scatter", mode="ez", storage=case["storage"], streaming="two_buffers", source="line", nx=n, ny=n,
                 nz=1, width=8 if n < 128 else 16, wavelength=rng.randint(8, 16) if small else rng.randint(24, 48))
            for n in (32 * -(-rng.randint(case["lo"], case["hi"]) // 32) for _ in range(case["count"]))]


# --------------------------------------------------------- prepare and run
def _solver(case, seed):
    s = lbem.Solver((case["nx"], case["ny"], case["nz"]), _eps(case, seed), mode=case["mode"], storage=case["storage"],
                    absorber_width=case["width"], sigma_max=SIGMA_MAX, streaming=case["streaming"])
    s.inject(_wave(case))
    return s


def prepare(case, seed):
    if case["kind"] == "adjoint":
        T = _period(case)
        problem = SimpleNamespace(mode=case["mode"], absorber_width=case["width"], sigma_max=SIGMA_MAX,
                                  wave=_wave(case), steps=case["steps"], dft_start=case["steps"] - T + 1,
                                  dft_periods=1)
        theta = np.linspace(0.0, math.pi / 2, case["angles"])
        return SimpleNamespace(kind="adjoint", eps=_eps(case, seed).requires_grad_(True), problem=problem, theta=theta,
                               phi=np.zeros_like(theta) if case["mode"] == "3d" else None, every=case["every"])
    if case["kind"] == "batch":
        cases = _batch_cases(case)
        solvers = [_solver(c, seed + k) for k, c in enumerate(cases)]
        batch = lbem.Batch(solvers)
        batch.run([_warm(c) for c in cases])
        cells = sum(c["nx"] * c["ny"] for c in cases)
        E, H = (torch.empty(3 * cells, dtype=torch.float32, device="cuda") for _ in range(2))
        return SimpleNamespace(kind="batch", solvers=solvers, batch=batch, periods=[_period(c) for c in cases], E=E, H=H,
                               theta=_angles("ez")[0])
    s = _solver(case, seed)
    s.step(_warm(case))
    E, H = (torch.empty((3, case["nz"], case["ny"], case["nx"]), dtype=torch.float32, device="cuda") for _ in range(2))
    theta, phi = _angles(case["mode"])
    return SimpleNamespace(kind="scatter", solver=s, period=_period(case), E=E, H=H, theta=theta, phi=phi,
                           far=case["source"] == "line")


def run(state):
    if state.kind == "adjoint":
        state.eps.grad = None
        s2 = far_field_intensity(state.eps, state.problem, state.theta, state.phi, state.every)
        s2.sum().backward()
        return dict(s2=s2.detach(), grad=state.eps.grad)
    if state.kind == "batch":
        for s, T in zip(state.solvers, state.periods):
            s.set_dft_window(s.time + 1, 1)
        state.batch.run(state.periods)
        s2 = [s.far_field(state.theta) for s in state.solvers]
        at = 0
        for s in state.solvers:
            n = 3 * s.shape[0] * s.shape[1]
            lbem.lbem_fields(s.h, state.E[at:at + n], state.H[at:at + n])
            at += n
        return dict(s2=np.concatenate(s2), E=state.E, H=state.H)
    s = state.solver
    out = {}
    if state.far:
        s.set_dft_window(s.time + 1, 1)
    s.step(state.period)
    if state.far:
        out["s2"] = s.far_field(state.theta, state.phi)
    out["energy"] = s.energy()
    lbem.lbem_fields(s.h, state.E, state.H)
    return dict(out, E=state.E, H=state.H)


# ------------------------------------------------------------------- work
def work(case):
    """Bytes: the state in and out once, the permittivity, the field maps and
    far-field inputs; a gradient reads eps and writes it once.  Flops: the
    update's own additions and products (21 or 42 populations: moments, fields,
    equilibria, collision), for a gradient those of the transposed update too."""
    if case["kind"] == "batch":
        parts = [work(c) for c in _batch_cases(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    cells = case["nx"] * case["ny"] * case["nz"]
    Q, per = (42, 123) if case["mode"] == "3d" else (21, 58)
    if case["kind"] == "adjoint":
        return dict(bytes=8.0 * cells, flops=2.0 * per * cells * case["steps"])
    return dict(bytes=cells * (2.0 * Q * (4 if case["storage"] == "f32" else 2) + 4 + 24),
                flops=float(per) * cells * _period(case))


# ------------------------------------------------------- FP64 in plain torch
# velocities 0, +x, -x, +y, -y, +z, -z
_VEL = ((0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1))
_COMPS = {"ez": ((2,), (0, 1)), "hz": ((0, 1), (2,)), "3d": ((0, 1, 2), (0, 1, 2))}


def _cross(c, V):
    """c x V for a component dict V (missing components are zero)."""
    out = {}
    for a in range(3):
        terms = [s * V[k] for s, k in ((c[(a + 1) % 3], (a + 2) % 3), (-c[(a + 2) % 3], (a + 1) % 3))
                 if s != 0 and k in V]
        if terms:
            out[a] = sum(terms)
    return out


def _equilibrium(i, E, H, eps, a, fam):
    """Component a of e_i (fam 0) or h_i (fam 1) in equilibrium with (E, H)."""
    if i == 0:
        return (eps - 1.0) * E[a] if fam == 0 else 0.0 * H[a]
    if fam == 0:
        return (E[a] - _cross(_VEL[i], H).get(a, 0.0)) / 6.0
    return (H[a] + _cross(_VEL[i], E).get(a, 0.0)) / 6.0


class _Lattice:
    """FP64 populations f[i][c][z][y][x], c over the mode's e then h components."""

    def __init__(self, mode, eps, width):
        self.mode, self.eps = mode, eps
        self.ec, self.hc = _COMPS[mode]
        nz, ny, nx = eps.shape
        d = None
        for m, shape in ((nx, (1, 1, -1)), (ny, (1, -1, 1)), (nz, (-1, 1, 1))):
            if m == 1:
                continue
            k = torch.arange(m, device=eps.device, dtype=torch.float64)
            k = torch.minimum(k, m - 1 - k).reshape(shape)
            d = k if d is None else torch.minimum(d, k)
        depth = torch.clamp(width - d, min=0.0) / max(1, width)
        self.keep = 1.0 - SIGMA_MAX * depth ** 3
        self.f = torch.zeros((7, len(self.ec) + len(self.hc), nz, ny, nx), dtype=torch.float64, device=eps.device)

    def pulled(self, f):
        out = []
        for i, c in enumerate(_VEL):
            g = f[i]
            for ax, dim in ((0, 3), (1, 2), (2, 1)):
                n = g.shape[dim]
                if c[ax] > 0 and n > 1:
                    g = torch.cat([g.narrow(dim, 0, 1), g.narrow(dim, 0, n - 1)], dim)
                elif c[ax] < 0 and n > 1:
                    g = torch.cat([g.narrow(dim, 1, n - 1), g.narrow(dim, n - 1, 1)], dim)
            out.append(g if i and g is not f[i] else g.clone())
        return out

    def moments(self, u):
        m = u[0]
        for i in range(1, 7):
            m = m + u[i]
        E = {a: m[k] / self.eps for k, a in enumerate(self.ec)}
        H = {a: m[len(self.ec) + k] for k, a in enumerate(self.hc)}
        return E, H

    def collided(self, u, E, H):
        f = []
        for i in range(7):
            eq = [_equilibrium(i, E, H, self.eps, a, 0) for a in self.ec]
            eq += [_equilibrium(i, E, H, self.eps, a, 1) for a in self.hc]
            f.append(self.keep * (2.0 * torch.stack(eq) - u[i]))
        return torch.stack(f)


class _Run:
    """A whole run: lattice, incident line or closed-form wave, DFT of the near fields."""

    def __init__(self, case, eps, t_window):
        self.case, self.w, self.T = case, _wave(case), _period(case)
        self.main = _Lattice(case["mode"], eps, case["width"])
        self.n = (case["nx"], case["ny"], case["nz"])
        self.t, self.t0 = 0, t_window
        self.X, self.line_X = None, None
        self.axis = [k for k in range(3) if abs(self.w.direction[k]) == 1.0]
        if self.axis:
            self.axis = self.axis[0]
            shape = [1, 1, 1]
            shape[2 - self.axis] = self.n[self.axis]
            self.line = _Lattice(case["mode"], torch.ones(shape, dtype=torch.float64, device=eps.device), case["width"])
        else:
            self.line = None

    def _fields_at(self, s):
        d, p = self.w.direction, self.w.polarization
        q = (d[1] * p[2] - d[2] * p[1], d[2] * p[0] - d[0] * p[2], d[0] * p[1] - d[1] * p[0])
        return {a: s * p[a] for a in self.main.ec}, {a: s * q[a] for a in self.main.hc}

    def _ramped(self, tau):
        tr = self.w.ramp_periods * self.T
        ramp = torch.where(tau <= 0, 0.0, torch.where(tau >= tr, 1.0, 0.5 * (1 - torch.cos(math.pi * tau / tr))))
        return self.w.amplitude * ramp * torch.sin(2 * math.pi / self.T * tau)

    def _incident(self, i, box):
        """Incident populations of direction i on the cells of box = ((x0, x1), (y0, y1), (z0, z1)) at time t."""
        if self.line is not None:
            idx = [slice(None)] * 4
            idx[3 - self.axis] = slice(*box[self.axis])
            return self.line.f[i][tuple(idx)]
        dev = self.main.eps.device
        x, y, z = (torch.arange(*b, device=dev, dtype=torch.float64) for b in box)
        k, r0 = self.w.direction, self.w.origin
        proj = (k[0] * (x - r0[0]))[None, None, :] + (k[1] * (y - r0[1]))[None, :, None] + \
            (k[2] * (z - r0[2]))[:, None, None]
        E, H = self._fields_at(self._ramped(self.t - 3.0 * proj))
        return torch.stack([_equilibrium(i, E, H, 1.0, a, 0) for a in self.main.ec] +
                           [_equilibrium(i, E, H, 1.0, a, 1) for a in self.main.hc])

    def _links(self, u):
        """The incident population of the link's source cell, added on links into the total-field box, removed on links out of it."""
        lo = self.w.tf_lo
        hi = [min(h, m - 1) for h, m in zip(self.w.tf_hi, self.n)]
        for i in range(1, 7):
            ax = (i - 1) // 2
            if self.n[ax] == 1:
                continue
            step = _VEL[i][ax]
            for into in (True, False):
                first, last = (lo[ax], hi[ax]) if step > 0 else (hi[ax], lo[ax])
                src = first - step if into else last
                dst = src + step
                if not (0 <= src < self.n[ax] and 0 <= dst < self.n[ax]):
                    continue
                box = [[lo[k], hi[k] + 1] for k in range(3)]
                box[ax] = [src, src + 1]
                inc = self._incident(i, box)
                box[ax] = [dst, dst + 1]
                cells = u[i][:, box[2][0]:box[2][1], box[1][0]:box[1][1], box[0][0]:box[0][1]]
                cells += inc if into else -inc

    def _faces(self, E, H):
        got = []
        for ax in range(3):
            if self.n[ax] == 1:
                continue
            for side in (0, 1):
                idx = [slice(self.w.ntff_lo[k], self.w.ntff_hi[k] + 1) for k in (2, 1, 0)]
                idx[2 - ax] = (self.w.ntff_lo, self.w.ntff_hi)[side][ax]
                idx = tuple(idx)
                got.append(torch.stack([E[a][idx] for a in self.main.ec] + [H[a][idx] for a in self.main.hc]))
        return got

    def step(self, f):
        t = self.t + 1
        u = self.main.pulled(f)
        self._links(u)
        E, H = self.main.moments(u)
        recorded = None
        window = self.t0 is not None and self.t0 <= t < self.t0 + self.T
        coef = None
        if window:
            ph = 2 * math.pi * (t % self.T) / self.T
            coef = 2.0 / self.T * complex(math.cos(ph), -math.sin(ph))
            recorded = [v * coef for v in self._faces(E, H)]
        f = self.main.collided(u, E, H)
        if self.line is not None:
            lu = self.line.pulled(self.line.f)
            lE, lH = self.line.moments(lu)
            if window:
                pol = self.w.polarization
                e = sum(pol[a] * lE[a].reshape(-1) for a in self.main.ec) * coef
                self.line_X = e if self.line_X is None else self.line_X + e
            g = self.line.collided(lu, lE, lH)
            s = self._ramped(torch.tensor(float(t), dtype=torch.float64))
            sE, sH = self._fields_at(float(s))
            idx = [slice(None)] * 3
            idx[2 - self.axis] = self.w.source_index
            for i in range(7):
                for k, a in enumerate(self.main.ec + self.main.hc):
                    fam = 0 if k < len(self.main.ec) else 1
                    g[(i, k) + tuple(idx)] = _equilibrium(i, sE, sH, 1.0, a, fam)
            self.line.f = g
        self.t = t
        return f, recorded

    def advance(self, f, steps):
        """f after `steps` steps, and the sums of what the DFT window recorded in them."""
        X = None
        for _ in range(steps):
            f, rec = self.step(f)
            if rec is not None:
                X = rec if X is None else [p + q for p, q in zip(X, rec)]
        return f, X

    def intensity(self, X, theta, phi):
        w, mode, dev = self.w, self.case["mode"], self.main.eps.device
        k = 2 * math.pi / w.wavelength
        c = w.center[self.axis]
        i0 = int(math.floor(c))
        ei = 0.5 * sum(abs(complex(self.line_X[min(i, self.n[self.axis] - 1)])) for i in (i0, i0 + 1))
        th = torch.as_tensor(theta, dtype=torch.float64, device=dev)
        zero = torch.zeros_like(th)
        if mode == "3d":
            ph = torch.as_tensor(phi, dtype=torch.float64, device=dev)
            rhat = (th.sin() * ph.cos(), th.sin() * ph.sin(), th.cos())
            tv, pv = (th.cos() * ph.cos(), th.cos() * ph.sin(), -th.sin()), (-ph.sin(), ph.cos(), zero)
        else:
            rhat, pv = (th.cos(), th.sin(), zero), (-th.sin(), th.cos(), zero)
        N, L = [0.0] * 3, [0.0] * 3
        at = 0
        for ax in range(3):
            if self.n[ax] == 1:
                continue
            for side in (0, 1):
                face = X[at]
                at += 1
                E = {a: face[j] for j, a in enumerate(self.main.ec)}
                H = {a: face[len(self.main.ec) + j] for j, a in enumerate(self.main.hc)}
                normal = [0, 0, 0]
                normal[ax] = 1 if side else -1
                J, M = _cross(normal, H), {a: -v for a, v in _cross(normal, E).items()}
                fac = []
                for b in (2, 1, 0):
                    if b == ax:
                        continue
                    p = torch.arange(w.ntff_lo[b], w.ntff_hi[b] + 1, device=dev, dtype=torch.float64)
                    wt = torch.ones_like(p)
                    if len(p) > 1:
                        wt[0] = wt[-1] = 0.5
                    fac.append(torch.exp(1j * k * rhat[b][:, None] * (p - w.center[b])) * wt)
                pw = torch.exp(1j * k * rhat[ax] * ((w.ntff_lo, w.ntff_hi)[side][ax] - w.center[ax]))
                for got, V in ((N, J), (L, M)):
                    for a, v in V.items():
                        got[a] = got[a] + pw * ((fac[0] @ v.reshape(fac[0].shape[1], -1)) * fac[1]).sum(1)
        dot = lambda u, V: sum(x * y for x, y in zip(u, V))  # noqa: E731
        if mode == "3d":
            a1, a2 = dot(tv, N) + dot(pv, L), dot(pv, N) - dot(tv, L)
            return k ** 4 * (a1.abs() ** 2 + a2.abs() ** 2) / (16 * math.pi ** 2 * ei ** 2)
        a = N[2] - dot(pv, L) if mode == "ez" else dot(pv, N) + L[2]
        return k * k * a.abs() ** 2 / (8 * math.pi * ei ** 2)


def _exact_scatter(case, seed):
    eps = _eps(case, seed).double()
    warm, T = _warm(case), _period(case)
    r = _Run(case, eps, warm + 1 if case["source"] == "line" else None)
    f, X = r.advance(r.main.f, warm + T)
    E, H = r.main.moments(f)
    energy = 0.5 * (sum((eps * v * v).sum() for v in E.values()) + sum((v * v).sum() for v in H.values()))
    zero = torch.zeros_like(eps)
    out = {}
    if X is not None:
        out["s2"] = r.intensity(X, *_angles(case["mode"])).cpu().numpy()
    return dict(out, energy=float(energy), E=torch.stack([E.get(a, zero) for a in range(3)]),
                H=torch.stack([H.get(a, zero) for a in range(3)]))


def _exact_adjoint(case, seed):
    eps = _eps(case, seed).double().requires_grad_(True)
    r = _Run(case, eps.detach(), case["steps"] - _period(case) + 1)
    theta = np.linspace(0.0, math.pi / 2, case["angles"])
    phi = np.zeros_like(theta) if case["mode"] == "3d" else None
    seg = 15 if case["mode"] == "3d" else 40
    starts, lines, f = [], [], r.main.f
    parts = []
    with torch.no_grad():
        while r.t < case["steps"]:
            starts.append((r.t, f))
            lines.append((r.line.f, r.line_X))
            f, X = r.advance(f, min(seg, case["steps"] - r.t))
            parts.append(X)
    Xs = [p for p in parts if p is not None]
    total = [sum(v).detach().requires_grad_(True) for v in zip(*Xs)]
    s2 = r.intensity(total, theta, phi)
    s2.sum().backward()
    gX = [x.grad for x in total]
    grad, gf = torch.zeros_like(eps), torch.zeros_like(f)
    for (t, f0), (line, line_X), X in zip(reversed(starts), reversed(lines), reversed(parts)):
        e = eps.detach().clone().requires_grad_(True)
        r.main.eps = e
        r.t, r.line.f, r.line_X = t, line, line_X
        f0 = f0.detach().clone().requires_grad_(True)
        f1, X1 = r.advance(f0, min(seg, case["steps"] - t))
        outs, grads = [f1], [gf]
        if X1 is not None:
            outs, grads = outs + X1, grads + gX
        gf, ge = torch.autograd.grad(outs, [f0, e], grads)
        grad += ge
    return dict(s2=s2.detach(), grad=grad)


def exact(case, seed):
    """FP64 values of run's outputs from a new state; None where it would take too long."""
    if case["kind"] == "batch":
        return None
    values = case["nx"] * case["ny"] * case["nz"] * (42 if case["mode"] == "3d" else 21)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed) if values * case["steps"] < 2.5e10 and case["steps"] <= 4000 else None
    return _exact_scatter(case, seed) if values * (_warm(case) + _period(case)) < 1.5e11 else None
