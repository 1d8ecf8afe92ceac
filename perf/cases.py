"""Performance cases of the particle step: what a user of the framework has it do.

Each case is one call pattern of the public entry points (paper_2101_02745_gb300.emu,
.adjoint) at one size: classic RK4 steps of single boxes from the smallest run to the
throughput box, with each shape order and the vacuum and matter terms, a batched
parameter sweep, gradients through the run, 3D boxes, particles off the lattice, and
the field outputs an analysis reads.  `exact` restates the equations (Eq. 2, 4-9 of
arXiv:2101.02745) in plain torch and numpy, in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2101_02745_gb300 import emu as E
from paper_2101_02745_gb300 import workloads as W
from paper_2101_02745_gb300.adjoint import Evolve, Simulation

DEV = "cuda:0"
# three-flavour vacuum and matter terms comparable to the self-interaction, every angle and the phase on
OSC = dict(mass_eV=(0.01, 0.02, 0.05), theta12=0.59, theta13=0.15, theta23=0.84, delta_cp=1.0,
           energy_MeV=5e-5, rho_g_cm3=1e8, Ye=0.4)


def _case(name, kind, nz, ndir, steps=1, order=2, osc=False, alpha=1e-6, nx=1, ny=1, nbox=1, fiducial=False):
    """alpha is the perturbation of Eq. 9: 1e-6 starts the run (its linear phase), 0.3 stands
    for a run past saturation, where every component of the density matrices is of order one."""
    return dict(name=name, kind=kind, nz=nz, ndir=ndir, steps=steps, order=order, osc=osc, alpha=alpha, nx=nx, ny=ny,
                nbox=nbox, fiducial=fiducial)


def listed():
    return [
        # the smallest run: the fiducial 32-cell box, ten steps a call between outputs
        _case("fiducial_32x16", "step", 32, 16, steps=10, fiducial=True),
        # the growth-phase box of the gradient study, stepped
        _case("growth_256x96", "step", 256, 96, steps=4, fiducial=True),
        # the paper's run shape (Sec. 3.1), past saturation
        _case("paper_1024x378", "step", 1024, 378, steps=2, alpha=0.3, fiducial=True),
        # production throughput box, per-cell densities and fluxes, at the start of a run
        _case("throughput_16384x1000", "step", 16384, 1000),
        # ragged box with the cubic shape and the vacuum and matter terms
        _case("cubic_osc_1999x251", "step", 1999, 251, order=3, osc=True, alpha=0.3),
        # ragged box with the linear shape (cloud in cell)
        _case("linear_777x130", "step", 777, 130, steps=2, order=1, alpha=0.3),
        # parameter sweep: uneven boxes advanced by the same launches (Sec. 4)
        _case("sweep_64_boxes", "sweep", 1024, 378, nbox=64),
        # gradients of the final moments' objectives through a run (forward and backward)
        _case("gradient_256x96", "gradient", 256, 96, steps=40, fiducial=True),
        # 3D box
        _case("box3d_64x64x64x16", "box3d", 64, 16, nx=64, ny=64),
        # particles off the lattice with a direction each, at the paper's run shape
        _case("anywhere_1024x378", "anywhere", 1024, 378, steps=2, alpha=0.3),
        # what an analysis reads from a snapshot: potential, Hamiltonians, moments, diagnostics
        _case("fields_2048x1000", "fields", 2048, 1000, alpha=0.3),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "step", "step", "step", "sweep", "gradient", "box3d", "anywhere", "fields"])
    alpha = rng.choice([1e-6, 0.3])
    fid = rng.random() < 0.3
    if kind == "step":
        nz, m = logint(30, 16384), logint(12, 1000)
        order = rng.choice([0, 1, 2, 2, 2, 3])
        # (one step with the delta shape: later stage positions can land on a cell face, where rounding decides)
        steps = 1 if order == 0 or nz * m >= 10**6 else 10 if nz * m < 4000 else 2
        return _case("", kind, nz, m, steps=steps, order=order, osc=rng.random() < 0.25, alpha=alpha, fiducial=fid)
    if kind == "sweep":
        return _case("", kind, logint(100, 1024), logint(60, 378), nbox=logint(4, 64), alpha=alpha)
    if kind == "gradient":
        return _case("", kind, logint(40, 256), logint(12, 96), steps=rng.randint(5, 40), fiducial=fid)
    if kind == "box3d":
        return _case("", kind, logint(12, 64), logint(6, 24), nx=logint(9, 64), ny=logint(9, 64),
                     order=rng.choice([1, 2, 2, 3]), alpha=alpha)
    if kind == "anywhere":
        return _case("", kind, logint(64, 1024), logint(24, 378), steps=2, order=rng.choice([1, 2, 2, 3]), alpha=alpha)
    return _case("", kind, logint(64, 2048), logint(24, 1000), order=rng.choice([1, 2, 2, 3]), alpha=alpha)


# ------------------------------------------------------------------ inputs

def _directions(M):
    """Midpoint Fibonacci sphere."""
    d = np.arange(M)
    mu = 1.0 - (2.0 * d + 1.0) / M
    phi = d * (math.pi * (3.0 - math.sqrt(5.0)))
    s = np.sqrt(1.0 - mu * mu)
    return np.stack([s * np.cos(phi), s * np.sin(phi), mu], axis=1)


def _species(case, C, rng):
    """Per-cell densities and fluxes of both species [cm^-3]: the fiducial ones with the
    densities of the seed within 10 %, or drawn per cell."""
    if case["fiducial"]:
        n = np.full(C, 4.9e32 * rng.uniform(0.9, 1.0))
        nb = np.full(C, 6.1e32 * rng.uniform(0.9, 1.0))
        f = np.zeros((C, 3))
        fb = np.zeros((C, 3))
        fb[:, 2] = -nb / 3.0
        return n, nb, f, fb
    n, nb = rng.uniform(1e32, 1e33, C), rng.uniform(1e32, 1e33, C)

    def flux(dens):
        v = rng.normal(size=(C, 3))
        v /= np.linalg.norm(v, axis=1, keepdims=True)
        return v * (rng.uniform(0.0, 0.33, C) * dens)[:, None]

    return n, nb, flux(n), flux(nb)


def _boxes(case, seed):
    """The plain numbers of each box of a case: sizes, inputs, step size."""
    rng, sizes = (np.random.Generator(np.random.PCG64(k)) for k in (seed, 0))   # (the sizes are the case's own)
    out = []
    for b in range(case["nbox"]):
        nz, M = case["nz"], case["ndir"]
        if case["nbox"] > 1:
            nz, M = int(sizes.integers(max(nz // 16, 1), nz + 1)), int(sizes.integers(max(M // 8, 1), M + 1))
        h = 13.42 / 32 if case["fiducial"] else 1.0 / 16.0
        C = case["nx"] * case["ny"] * nz
        n, nb, f, fb = _species(case, C, rng)
        osc = W.oscillation(**OSC) if case["osc"] else None
        top = max(float(n.max()), float(nb.max()), osc["n_e"] if osc else 0.0)
        dt = 0.4 * min(h / W.C_LIGHT, 1.0 / (W.KAPPA * top))
        out.append(dict(nx=case["nx"], ny=case["ny"], nz=nz, ndir=M, h=h, C=C, n=n, nb=nb, f=f, fb=fb, osc=osc, dt=dt,
                        dirs=_directions(M), seed=seed * 1000 + b))
    return out


def _workload(case, x):
    return W.Workload(case["kind"], x["nz"], x["ndir"], x["h"] * x["nz"], x["n"], x["nb"], x["f"], x["fb"],
                      dirs=x["dirs"], alpha=case["alpha"], seed=x["seed"], shape_order=case["order"])


def _scatter(x, seed):
    """Positions moved by up to 0.45 cells and a random direction per particle."""
    rng = np.random.Generator(np.random.PCG64([seed, 1]))
    P, Lz = x["C"] * x["ndir"], x["h"] * x["nz"]
    z = (np.tile(np.arange(x["nz"]) + 0.5, x["ndir"]) + rng.uniform(-0.45, 0.45, P)) * x["h"]
    om = rng.normal(size=(P, 3))
    om /= np.linalg.norm(om, axis=1, keepdims=True)
    return np.where(z >= Lz, z - Lz, z), om


def prepare(case, seed):
    xs = _boxes(case, seed)
    x, kind = xs[0], case["kind"]
    st = dict(kind=kind, steps=case["steps"], dt=x["dt"])
    if kind == "box3d":
        wl = W.Workload3("box3d", x["nx"], x["ny"], x["nz"], x["ndir"], x["nx"] * x["h"], x["ny"] * x["h"],
                         x["nz"] * x["h"], x["n"], x["nb"], x["f"], x["fb"], dirs=x["dirs"], alpha=case["alpha"],
                         seed=x["seed"], shape_order=case["order"])
        st["box"] = E.Box3D.from_workload(wl, device=DEV)
        return st
    if kind == "sweep":
        st["box"] = E.Box.from_workloads([_workload(case, v) for v in xs], device=DEV)
        st["box"].batch_set_dt(np.array([v["dt"] for v in xs]))
        return st
    st["box"] = box = E.Box.from_workload(_workload(case, x), device=DEV, init=kind != "gradient")
    if case["osc"]:
        box.set_oscillation(x["osc"])
    if kind == "anywhere":
        z, om = _scatter(x, seed)
        box.set_host(z=z, ox=om[:, 0].copy(), oy=om[:, 1].copy(), oz=om[:, 2].copy())
    if kind == "gradient":
        st["inputs"] = [torch.tensor(a, device=DEV, requires_grad=True) for a in (x["n"], x["nb"], x["f"], x["fb"])]
        st["sim"] = Simulation(box, case["steps"], x["dt"], every=20, alpha=case["alpha"], seed=x["seed"],
                               dirs=x["dirs"])
    return st


def _loss(mom):
    """Mean nu_e abundance and the growth measure <|n_emu|> (Eq. 10), of one size."""
    return mom[0].mean() / 1e32 + torch.log(torch.hypot(mom[3], mom[4]).mean())


def run(state):
    box, kind = state["box"], state["kind"]
    if kind == "gradient":
        mom = Evolve.apply(*state["inputs"], state["sim"])
        grads = torch.autograd.grad(_loss(mom), state["inputs"])
        return {"moments": mom.detach(), "dn": grads[0], "dnbar": grads[1], "df": grads[2], "dfbar": grads[3]}
    if kind == "fields":
        return {"potential": box.deposit(), "H": box.interpolate_H(), "moments": box.moments(),
                "diagnostics": box.diagnostics()}
    if kind == "sweep":
        box.batch_step(state["steps"])
    else:
        box.step(state["steps"], state["dt"])
    return {k: box.t[k] for k in (("x", "y", "z") if kind == "box3d" else ("z",)) + ("rho", "rhobar")}


def work(case):
    """Each particle's position, direction, weights and matrices read once and what the call
    changes or returns written once; the equations' floating-point operations."""
    reach = {0: 1, 1: 2, 2: 3, 3: 4}[case["order"]]
    taps = reach ** (3 if case["kind"] == "box3d" else 1)
    P = sum(x["C"] * x["ndir"] for x in _boxes(case, 0))
    C = sum(x["C"] for x in _boxes(case, 0))
    # per stage: B (27), its spread (2 taps a real) and four moments (56), A0 - Omega . A (48),
    # interpolation (2 taps a real), two commutators (168), RK4 update (72)
    stage = 27 + 56 + 48 + 168 + 72 + 2 * 8 * taps * 2
    nread = 26 if case["kind"] == "box3d" else 24
    if case["kind"] == "fields":
        # the snapshot read once; potential, H, moments and diagnostics written
        return {"bytes": 8.0 * (24 * P + 9 * P + 108 * C + 63), "flops": float(P) * (3 * 9 * (2 * taps + 8) + 27 + 72)}
    if case["kind"] == "gradient":
        # inputs and moments; a step forward and its transpose (twice the forward's operations)
        return {"bytes": 8.0 * (8 * C * 2 + 72 * C), "flops": 3.0 * 4 * stage * P * case["steps"]}
    return {"bytes": 8.0 * (nread + nread - 5) * P, "flops": 4.0 * stage * P * case["steps"]}


# ---------------------------------------------- the equations in plain torch

_PAIRS = ((0, 1, 3), (0, 2, 5), (1, 2, 7))


def _uniform(seed, k):
    """SplitMix64 output k + 1 of the stream `seed`, as a number in [-1, 1)."""
    with np.errstate(over="ignore"):
        s = np.uint64(seed) + (k + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        s = (s ^ (s >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        s = (s ^ (s >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        s = s ^ (s >> np.uint64(31))
    return 2.0 * ((s >> np.uint64(11)).astype(np.float64) * 2.0 ** -53) - 1.0


def _matrices(x, alpha):
    """Initial density matrices of Eq. 9, packed (9, P) per species."""
    p = np.arange(x["C"] * x["ndir"], dtype=np.uint64) * np.uint64(8)
    out = []
    for which in (0, 1):
        u = [alpha * _uniform(x["seed"], p + np.uint64(4 * which + k)) for k in range(4)]
        em, et = u[0] ** 2 + u[1] ** 2, u[2] ** 2 + u[3] ** 2
        zero = np.zeros_like(em)
        out.append(torch.tensor(np.stack([1.0 - em - et, em, et, *u, zero, zero]), device=DEV))
    return out


def _positions(x, ax):
    """Cell-centre coordinate along axis ax (0: x, 1: y, 2: z) of every particle."""
    n = (x["nx"], x["ny"], x["nz"])
    idx = torch.arange(x["C"], device=DEV, dtype=torch.float64)
    j = {2: idx % n[2], 1: torch.floor(idx / n[2]) % n[1], 0: torch.floor(idx / (n[2] * n[1]))}[ax]
    return ((j + 0.5) * x["h"]).repeat(x["ndir"])


def _bspline(order, t):
    """Centred cardinal B-spline of degree `order` at distance |t| cells."""
    t = t.abs()
    zero = torch.zeros_like(t)
    if order == 1:
        return torch.clamp(1.0 - t, min=0.0)
    if order == 2:
        return torch.where(t < 0.5, 0.75 - t * t, torch.where(t < 1.5, 0.5 * (1.5 - t) ** 2, zero))
    return torch.where(t < 1.0, 2.0 / 3.0 - t * t + 0.5 * t ** 3,
                       torch.where(t < 2.0, (2.0 - t) ** 3 / 6.0, zero))


def _stencil(order, pos, ncells, h):
    """[(cell index, weight)] of every cell a particle reaches along each axis, combined."""
    out = None
    for q, n in zip(pos, ncells):
        s = q / h
        base = torch.floor(s)
        reach = {0: (0,), 1: (-1, 0, 1), 2: (-1, 0, 1), 3: (-2, -1, 0, 1, 2)}[order]
        taps = []
        for o in reach:
            w = None if order == 0 else _bspline(order, s - (base + (o + 0.5)))
            taps.append((torch.remainder(base + o, n).long(), w))
        if out is None:
            out = taps
        else:
            out = [(c * n + c1, w1 if w is None else w * w1) for c, w in out for c1, w1 in taps]
    return out


def _unpack(v):
    m = [[None] * 3 for _ in range(3)]
    for a in range(3):
        m[a][a] = torch.complex(v[a], torch.zeros_like(v[a]))
    for a, b, k in _PAIRS:
        m[a][b] = torch.complex(v[k], v[k + 1])
        m[b][a] = m[a][b].conj()
    return m


def _commutator(H, r):
    """-i [H, r] packed; H and r as 3 x 3 lists of complex tensors."""
    def entry(a, b):
        c = sum(H[a][k] * r[k][b] - r[a][k] * H[k][b] for k in range(3))
        return c.imag, -c.real
    out = [entry(a, a)[0] for a in range(3)]
    for a, b, _ in _PAIRS:
        out += list(entry(a, b))
    return torch.stack(out)


_CONJ = (1, 1, 1, 1, -1, 1, -1, 1, -1)


def _vacuum_matter(osc):
    """Packed H_vacuum / hbar and H_matter / hbar of Eq. 2."""
    s12, c12 = math.sin(osc["theta12"]), math.cos(osc["theta12"])
    s13, c13 = math.sin(osc["theta13"]), math.cos(osc["theta13"])
    s23, c23 = math.sin(osc["theta23"]), math.cos(osc["theta23"])
    ep = complex(math.cos(osc["delta_cp"]), math.sin(osc["delta_cp"]))
    U = np.array([[c12 * c13, s12 * c13, s13 * ep.conjugate()],
                  [-s12 * c23 - c12 * s23 * s13 * ep, c12 * c23 - s12 * s23 * s13 * ep, s23 * c13],
                  [s12 * s23 - c12 * c23 * s13 * ep, -c12 * s23 - s12 * c23 * s13 * ep, c23 * c13]])
    w = (np.array(osc["mass_eV"]) * osc["erg_per_eV"]) ** 2 / (2.0 * osc["energy_erg"]) / osc["hbar"]
    H = (U * w) @ U.conj().T
    vac = [H[a, a].real for a in range(3)] + [f(H[a, b]) for a, b, _ in _PAIRS for f in (np.real, np.imag)]
    return [float(v) for v in vac], [W.KAPPA * osc["n_e"]] + [0.0] * 8


class _Exact:
    def __init__(self, case, x, n=None, nb=None, f=None, fb=None, pos=None, om=None):
        self.case, self.x, self.order = case, x, case["order"]
        self.axes = (0, 1, 2) if case["kind"] == "box3d" else (2,)
        self.ncells = [(x["nx"], x["ny"], x["nz"])[a] for a in self.axes]
        self.pos = [_positions(x, a) for a in self.axes] if pos is None else pos
        own = torch.tensor(x["dirs"], device=DEV)
        cols = [own[:, i].repeat_interleave(x["C"]) for i in range(3)]
        t = [torch.tensor(x[k], device=DEV) if v is None else v for k, v in
             (("n", n), ("nb", nb), ("f", f), ("fb", fb))]
        self.dV = x["h"] ** 3 if len(self.axes) == 3 else x["h"]

        def weight(dens, flux):
            fo = sum(flux[:, i].repeat(x["ndir"]) * cols[i] for i in range(3))
            return (dens.repeat(x["ndir"]) + 3.0 * fo) * (self.dV / x["ndir"])

        self.N, self.Nb = weight(t[0], t[2]), weight(t[1], t[3])
        self.om = cols if om is None else om
        self.r, self.rb = _matrices(x, case["alpha"])
        self.vac = _vacuum_matter(x["osc"]) if x["osc"] else None

    def spread(self, pos, B):
        """Sum of weight x (1, Omega) x B over particles, per cell: four (C, k) tensors."""
        out = [torch.zeros(self.x["C"], B.shape[0], dtype=torch.float64, device=DEV) for _ in range(4)]
        for m in range(4):
            v = B.T if m == 0 else (B * self.om[m - 1]).T
            for c, w in _stencil(self.order, pos, self.ncells, self.x["h"]):
                out[m] = out[m].index_add(0, c, v if w is None else w[:, None] * v)
        return out

    def hamiltonian(self, pos, A):
        H = None
        for c, w in _stencil(self.order, pos, self.ncells, self.x["h"]):
            for m in range(4):
                g = A[m][c].T if m == 0 else -A[m][c].T * self.om[m - 1]
                g = g if w is None else g * w
                H = g if H is None else H + g
        return H

    def potential(self, pos, r, rb):
        conj = torch.tensor(_CONJ, dtype=torch.float64, device=DEV)[:, None]
        return [a * (W.KAPPA / self.dV) for a in self.spread(pos, self.N * r - self.Nb * (conj * rb))]

    def rhs(self, shift, r, rb):
        pos = [q + shift * W.C_LIGHT * self.om[a] for q, a in zip(self.pos, self.axes)]
        H = self.hamiltonian(pos, self.potential(pos, r, rb))
        conj = torch.tensor(_CONJ, dtype=torch.float64, device=DEV)[:, None]
        Hb = -conj * H
        if self.vac:
            v, m = [torch.tensor(q, dtype=torch.float64, device=DEV)[:, None] for q in self.vac]
            H, Hb = H + v + m, Hb + conj * (v - m)
        return _commutator(_unpack(H), _unpack(r)), _commutator(_unpack(Hb), _unpack(rb))

    def step(self, dt):
        r, rb = self.r, self.rb
        acc, acb, sr, sb = r, rb, r, rb
        for frac, b, nxt in ((0.0, 6.0, 0.5), (0.5, 3.0, 0.5), (0.5, 3.0, 1.0), (1.0, 6.0, 0.0)):
            k, kb = self.rhs(frac * dt, sr, sb)
            acc, acb = acc + (dt / b) * k, acb + (dt / b) * kb
            sr, sb = r + (nxt * dt) * k, rb + (nxt * dt) * kb
        self.r, self.rb = acc, acb
        new = []
        for q, a, n in zip(self.pos, self.axes, self.ncells):
            L = n * self.x["h"]
            q = q + dt * W.C_LIGHT * self.om[a]
            q = torch.where(q >= L, q - L, torch.where(q < 0.0, q + L, q))
            new.append(q)
        self.pos = new

    def moments(self):
        return torch.cat([a.T / self.dV for B in (self.N * self.r, self.Nb * self.rb)
                          for a in self.spread(self.pos, B)])


def _diagnostics(mom):
    C = mom.shape[1]
    out = []
    for lo in (0, 36, 9, 45):
        v = mom[lo:lo + 9]
        mag = {(a, a): v[a].abs().mean() for a in range(3)}
        for a, b, k in _PAIRS:
            mag[a, b] = mag[b, a] = torch.hypot(v[k], v[k + 1]).mean()
        out += [mag[a, b] for a in range(3) for b in range(3)]
    conj = torch.tensor(_CONJ, dtype=torch.float64, device=mom.device)
    n, nb = mom[0:9].sum(1) / C, mom[36:45].sum(1) / C
    return torch.cat([torch.stack(out), n, nb, n - conj * nb]).cpu().numpy()


def exact(case, seed):
    xs, kind = _boxes(case, seed), case["kind"]
    x = xs[0]
    if kind == "gradient":
        t = [torch.tensor(x[k], device=DEV, requires_grad=True) for k in ("n", "nb", "f", "fb")]
        e = _Exact(case, x, *t)
        for _ in range(case["steps"]):
            e.step(x["dt"])
        mom = e.moments()
        g = torch.autograd.grad(_loss(mom), t)
        return {"moments": mom.detach(), "dn": g[0], "dnbar": g[1], "df": g[2], "dfbar": g[3]}
    parts = []
    for v in xs:
        if kind == "anywhere":
            z, om = _scatter(v, seed)
            e = _Exact(case, v, pos=[torch.tensor(z, device=DEV)],
                       om=[torch.tensor(om[:, i].copy(), device=DEV) for i in range(3)])
        else:
            e = _Exact(case, v)
        if kind == "fields":
            A = e.potential(e.pos, e.r, e.rb)
            mom = e.moments()
            return {"potential": torch.cat([a.T for a in A]), "H": e.hamiltonian(e.pos, A), "moments": mom,
                    "diagnostics": _diagnostics(mom)}
        for _ in range(case["steps"]):
            e.step(v["dt"])
        parts.append({**dict(zip("xyz" if kind == "box3d" else "z", e.pos)), "rho": e.r, "rhobar": e.rb})
    return {k: torch.cat([p[k] for p in parts], dim=-1) for k in parts[0]}
