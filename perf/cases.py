"""The work a user of this library has it do, as cases that can be timed and checked.

Every case is a call sequence of the public interface: a single lattice stepped
between two looks at its state (``Lattice.step`` and ``get`` / ``diag``), an
ensemble of runs (``Ensemble.step``), a training step and a prediction of the
surrogate (``Surrogate.train_step`` / ``predict``).  ``listed`` names the cases,
``draw`` gives more of the same ranges, ``prepare`` builds what the user holds
before the call, ``run`` is one pass, ``work`` the traffic and arithmetic a pass
cannot do without, and ``exact`` the same outputs in plain 64-bit torch.

Parameters are those of the repository's workloads (``synth.BASE``: b = 1,
kappa = -0.025, c = 0.02, Gamma = 0.05, Tc = 1) or of the paper's runs (b = 0.1,
kappa = -c = -0.03, Gamma = 0.1, Tc = 0.005).  Wall and initial temperatures are
given in units of Tc.  The compact stencils run with T_w = 0.9 Tc (the paper's
quench), the isotropic ones with 0.5 Tc: a lattice is stepped on from pass to
pass, and these stay finite however long they run.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1102_3094_gb300 import lf

PHYSICS = {
    "config": dict(b=1.0, kappa=-0.025, c=0.02, Gamma=0.05, Tc=1.0, phi_amp=0.05),
    "paper": dict(b=0.1, kappa=-0.03, c=0.03, Gamma=0.1, Tc=0.005, phi_amp=0.01),
}
ENS_SIZES = (128, 256, 384, 512)
ENS_TAUS = (0.6, 1.0, 3.0)
SUR_SCALE = (0.3, 0.2, 0.01, 0.01)      # spread of phi, T, ux, uy
SUR_OFFSET = (0.0, 0.9, 0.0, 0.0)


def _lattice(**kw):
    """A single-lattice case; what is not given is the default of the workloads."""
    c = dict(kind="lattice", d=2, nx=64, ny=64, nz=1, precision="fp32", stencil="compact", physics="config",
             walls=1, t_mode=0, solver="explicit", hydro=1, xi=1e-3, tau=1.0, tw=0.9, t0=1.1, steps=100, report=0)
    c.update(kw)
    return c


def listed():
    return [
        # The reference case: a 64 x 64 FP64 quench, diagnostics every 200 steps.  Launches and latency are all of it.
        _lattice(name="report64", nx=64, ny=64, precision="fp64", xi=0.01, steps=200, report=1),
        # The paper's 2D lattice with its parameters and hydrodynamics (slow front), as the phenomenology runs step it.
        _lattice(name="paper256", nx=256, ny=256, physics="paper", xi=1e-4, tau=5.0, steps=300),
        # The precision form: 1024 x 1024 in FP32, looked at every 100 steps with its diagnostics.
        _lattice(name="prec1024", nx=1024, ny=1024, xi=1e-3, steps=100, report=1),
        # A large lattice whose sides fit no tile, a fast front (three temperature sub-steps), halfway thermal walls.
        _lattice(name="ragged2d", nx=2999, ny=1777, xi=0.5, t_mode=1, steps=20),
        # The isotropic stencils on the 1024 x 1024 fast-front run (the compact ones go non-finite there).
        _lattice(name="iso1024", nx=1024, ny=1024, stencil="isotropic", xi=0.1, tw=0.5, steps=100),
        # The paper's 3D run: 32 x 32 x 256, finite differences alone, xi = 1 (eight temperature sub-steps).
        _lattice(name="slab3d", d=3, nx=32, ny=32, nz=256, stencil="isotropic", physics="paper", hydro=0, xi=1.0,
                 steps=110),
        # The benchmark workload: 384^3 D3Q19 in FP32.
        _lattice(name="cube384", d=3, nx=384, ny=384, nz=384, xi=1e-3, tau=0.6, steps=10),
        # The 3D configuration that runs its full length (isotropic, tau = 3), on sides that fit no tile.
        _lattice(name="iso3d", d=3, nx=250, ny=243, nz=190, stencil="isotropic", xi=1e-2, tau=3.0, tw=0.5, steps=20),
        # A front too fast for explicit sub-steps: backward-Euler temperature on 256^3.
        _lattice(name="implicit256", d=3, nx=256, ny=256, nz=256, solver="implicit", xi=100.0, steps=4),
        # The batched sweep: 96 independent runs of four sizes, xi log-uniform, three relaxation times.
        dict(name="ens96", kind="ensemble", runs=96, stencil="compact", tw=0.9, steps=200),
        # One training step of the surrogate at the batch size its training uses, and the weights it gives.
        dict(name="train16", kind="train", batch=16, ny=256, nx=256, lr=1e-3),
        # One prediction for one lattice: what a surrogate window of an interleaved run costs.
        dict(name="predict1", kind="predict", batch=1, ny=256, nx=256),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _size(rng, lo, hi):
    """A lattice side, log-uniform: any integer, or (as often) the nearest multiple of 32."""
    n = int(round(_log(rng, lo, hi)))
    return n if rng.random() < 0.5 else max(32, 32 * round(n / 32))


def _steps(sites, per_step):
    """Steps between two looks at the state: fewer on larger lattices."""
    return max(2, min(300, int(per_step / sites)))


FFT_SIDES = (64, 90, 96, 100, 120, 125, 128, 144, 160, 162, 192, 200, 210, 240, 243, 250, 256)


def draw(rng):
    kind = rng.choice(["2d", "2d", "2d", "3d", "3d", "3d", "implicit", "ensemble", "train", "predict"])
    if kind == "ensemble":
        return dict(kind="ensemble", runs=rng.randrange(4, 97), stencil=rng.choice(["compact", "isotropic"]), tw=0.9,
                    steps=rng.randrange(20, 200))
    if kind in ("train", "predict"):
        c = dict(kind=kind, batch=rng.randrange(1, 17), ny=rng.randrange(64, 257), nx=rng.choice([128, 256]))
        if kind == "train":
            c["lr"] = round(_log(rng, 1e-5, 1e-3), 9)
        return c
    if kind == "implicit":
        if rng.random() < 0.5:
            nx, ny, nz, d = rng.choice(FFT_SIDES), rng.choice(FFT_SIDES), rng.randrange(40, 257), 3
        else:
            nx, ny, nz, d = rng.choice(FFT_SIDES) * rng.choice([1, 2, 4, 8]), _size(rng, 64, 2048), 1, 2
        return _lattice(d=d, nx=nx, ny=ny, nz=nz, solver="implicit", xi=round(_log(rng, 0.5, 100.0), 6),
                        t_mode=rng.randrange(2), steps=_steps(nx * ny * nz, 6.4e7))
    iso = rng.random() < 0.5
    c = dict(stencil="isotropic" if iso else "compact", walls=int(rng.random() < 0.8), t_mode=rng.randrange(2),
             hydro=int(rng.random() < 0.85), xi=round(_log(rng, 1e-4, 1.0), 9), report=int(rng.random() < 0.3))
    if kind == "2d":
        fp64 = rng.random() < 0.25
        nx, ny = _size(rng, 48, 1024 if fp64 else 4096), _size(rng, 48, 1024 if fp64 else 4096)
        c.update(nx=nx, ny=ny, precision="fp64" if fp64 else "fp32", tau=rng.choice([1.0, 3.0]),
                 steps=_steps(nx * ny, 2e7 if fp64 else 1.6e8))
        if c["report"]:                      # S(k) needs sides that the transform takes
            c.update(nx=rng.choice(FFT_SIDES) * rng.choice([1, 2, 4, 8]), ny=rng.choice(FFT_SIDES) * rng.choice([1, 2, 4]))
            c["steps"] = _steps(c["nx"] * c["ny"], 2e7 if fp64 else 1.6e8)
    else:
        nx, ny, nz = _size(rng, 24, 384), _size(rng, 24, 384), _size(rng, 24, 384)
        c.update(d=3, nx=nx, ny=ny, nz=nz, tau=3.0, steps=_steps(nx * ny * nz, 3e8), report=0)
    if iso:
        c["tw"] = 0.5 if c["walls"] else 0.9
    if not c["walls"]:
        c["t0"] = 0.9
    return _lattice(**c)


# ------------------------------------------------------------------ the calls
def _ens_members(case, seed):
    """Sizes in turn, xi log-uniform in [1e-4, 1], tau from the list: the library's ensemble workload."""
    rng = np.random.default_rng(seed)
    xis = 10.0 ** rng.uniform(-4.0, 0.0, size=case["runs"])
    taus = rng.choice(ENS_TAUS[1:] if case["stencil"] == "isotropic" else ENS_TAUS, size=case["runs"])
    return [dict(nx=ENS_SIZES[i % 4], ny=ENS_SIZES[i % 4], xi=float(xis[i]), tau=float(taus[i]), seed=seed * 1000 + i)
            for i in range(case["runs"])]


def _sur_fields(case, seed):
    """A batch of lamellar states (phi, T, ux, uy) and the states a little later, [B][4][NY][NX] FP32."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    B, NY, NX = case["batch"], case["ny"], case["nx"]

    def rnd(*shape):
        return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64) * 2 - 1

    y = torch.arange(NY, device="cuda", dtype=torch.float64).view(1, NY, 1)
    x = torch.arange(NX, device="cuda", dtype=torch.float64).view(1, 1, NX)
    out = []
    for shift in (0.0, 0.15):
        phase = 0.8 * y + 2 * math.pi * round(NX / 40) / NX * x + 3 * torch.arange(B, device="cuda").view(B, 1, 1) + shift
        phi = 0.4 * torch.cos(phase) + 0.05 * rnd(B, NY, NX)
        T = 0.9 + 0.2 * torch.tanh((y - NY / 2) / 20) * torch.ones_like(phi) + 0.01 * rnd(B, NY, NX)
        ux, uy = 0.01 * torch.sin(phase) + 0.002 * rnd(B, NY, NX), 0.01 * torch.cos(phase / 2) + 0.002 * rnd(B, NY, NX)
        out.append(torch.stack([phi, T, ux, uy], dim=1).float().contiguous())
    return out


SUR_LAYERS = ((16, 64), (64, 64), (64, 64), (64, 64), (64, 64), (64, 16))


def _sur_params(seed):
    """Network weights and biases, layer by layer ([9][cout][cin], then [cout]); the four input channels are used."""
    rng = np.random.default_rng(seed)
    parts = []
    for l, (cin, cout) in enumerate(SUR_LAYERS):
        lim = math.sqrt(6.0 / (9.0 * (4 if l == 0 else cin))) * (0.1 if l == 5 else 1.0)
        w = rng.uniform(-lim, lim, size=(9, cout, cin))
        if l == 0:
            w[:, :, 4:] = 0.0
        parts += [w.ravel(), rng.uniform(-0.02, 0.02, size=cout)]
    return np.concatenate(parts).astype(np.float32)


def _kwargs(case, seed):
    ph = PHYSICS[case["physics"]]
    return dict(ph, d=case["d"], nx=case["nx"], ny=case["ny"], nz=case["nz"], walls=case["walls"],
                t_wall_mode=case["t_mode"], T_w=case["tw"] * ph["Tc"], T0=case["t0"] * ph["Tc"], xi=case["xi"],
                tau=case["tau"], precision=case["precision"], hydro=case["hydro"], stencil=case["stencil"], seed=seed)


def prepare(case, seed):
    if case["kind"] == "lattice":
        sim = lf.Lattice(**_kwargs(case, seed))
        if case["solver"] == "implicit":
            sim.set_t_solver("implicit")
        return {"case": case, "sim": sim}
    if case["kind"] == "ensemble":
        members = _ens_members(case, seed)
        return {"case": case, "ens": lf.Ensemble(members, stencil=case["stencil"], T_w=case["tw"]), "n": len(members)}
    x, y = _sur_fields(case, seed)
    sur = lf.Surrogate(case["ny"], case["nx"], case["batch"], scale=SUR_SCALE, offset=SUR_OFFSET)
    sur.set_params(_sur_params(seed))
    return {"case": case, "sur": sur, "x": x, "y": y}


def run(state):
    case = state["case"]
    if case["kind"] == "lattice":
        sim, dt = state["sim"], case["precision"]
        sim.step(case["steps"])
        out = {k: sim.get(k, dtype=dt, device=True) for k in ("phi", "T", "pop")}
        if case["report"]:
            d = sim.diag()
            out["report"] = {k: d[k] for k in ("mass", "free_energy", "k_peak", "s_peak")}
            out["report"]["grad2"] = d["grad2"][:case["d"]]
        return out
    if case["kind"] == "ensemble":
        ens = state["ens"]
        ens.step(case["steps"])
        runs = [ens.run(r) for r in range(state["n"])]
        out = {}
        for i, n in enumerate(ENS_SIZES):
            if runs[i::4]:
                out[f"n{n}"] = {k: torch.stack([v.get(k, dtype="fp32", device=True) for v in runs[i::4]])
                                for k in ("phi", "T", "pop")}
        return out
    if case["kind"] == "train":
        loss = state["sur"].train_step(state["x"], state["y"], case["lr"])
        return {"loss": loss, "params": state["sur"].get_params()}
    return {"y": state["sur"].predict(state["x"])}


# ------------------------------------------------------------------ the floor
def work(case):
    """A lattice is read and written once per step (populations, phi, T; neither the populations without
    hydrodynamics nor anything between passes over the lattice), an implicit temperature once more, and the
    state that the user looks at is written once.  The network's inputs, outputs, weights and, in training,
    the activations that the backward pass needs in BF16 are moved once."""
    if case["kind"] in ("lattice", "ensemble"):
        if case["kind"] == "lattice":
            sites, d = case["nx"] * case["ny"] * case["nz"], case["d"]
            hydro, esz, impl = case["hydro"], 8 if case["precision"] == "fp64" else 4, case["solver"] == "implicit"
        else:
            sites = sum(ENS_SIZES[i % 4] ** 2 for i in range(case["runs"]))
            d, hydro, esz, impl = 2, 1, 4, False
        q = 9 if d == 2 else 19
        per = esz * (2 * (q if hydro else 0) + 4 + (2 if impl else 0))
        flops = (300 if d == 2 else 620) if hydro else 80
        return {"bytes": sites * (per * case["steps"] + esz * (q + 2)), "flops": sites * flops * case["steps"]}
    px = case["batch"] * case["ny"] * case["nx"]
    macs = sum(9 * cin * cout for cin, cout in SUR_LAYERS[1:5]) + 2 * 9 * 4 * 64
    if case["kind"] == "predict":
        return {"bytes": px * 32, "flops": 2 * macs * px}
    return {"bytes": px * (32 + 2 * 5 * 64 * 2), "flops": 3 * 2 * macs * px}


# ------------------------------------------------------------------ 64 bits
E2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
E3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
      (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]


def _weights(d):
    w = (4 / 9, 1 / 9, 1 / 36) if d == 2 else (1 / 3, 1 / 18, 1 / 36)
    return [w[sum(abs(c) for c in e)] for e in (E2 if d == 2 else E3)]


class _Exact:
    """A batch of lattices of one shape, [B][nz][ny][nx] (2D: [B][ny][nx]), in FP64; parameters may differ by run."""

    def __init__(self, d, walls, t_mode, stencil, hydro, phys, T_w, xi, tau, phi, T):
        self.d, self.walls, self.t_mode, self.iso, self.hydro, self.p = d, walls, t_mode, stencil == "isotropic", hydro, phys
        self.T_w, self.phi, self.T = T_w, phi, T
        shape = (phi.shape[0],) + (1,) * d
        self.xi = torch.tensor(xi, device=phi.device, dtype=torch.float64).view(shape)
        self.tau = torch.tensor(tau, device=phi.device, dtype=torch.float64).view(shape)
        self.nsub = [max(1, math.ceil(x / (0.8 / (2 * d)) - 1e-12)) for x in xi]
        self.E, self.w = (E2 if d == 2 else E3), _weights(d)
        self.f = [wi * torch.ones_like(phi) for wi in self.w]

    def nb(self, A, off, parity=1.0, ghost=None):
        """A(r + off); beyond a wall the mirror image times `parity`, or ghost - image."""
        for a in range(self.d - 1):
            if off[a]:
                A = torch.roll(A, -off[a], dims=-1 - a)
        o = off[self.d - 1]
        if not o:
            return A
        if not self.walls:
            return torch.roll(A, -o, dims=1)
        edge = A[:, -1:] if o > 0 else A[:, :1]
        edge = edge * parity if ghost is None else ghost - edge
        return torch.cat([A[:, 1:], edge] if o > 0 else [edge, A[:, :-1]], dim=1)

    def unit(self, a, s):
        return tuple(s if b == a else 0 for b in range(self.d))

    def lap(self, A, ghost=None):
        if self.iso:
            return sum(6 * wi * (self.nb(A, e, 1.0, ghost) - A) for e, wi in zip(self.E[1:], self.w[1:]))
        return sum(self.nb(A, self.unit(a, s), 1.0, ghost) - A for a in range(self.d) for s in (1, -1))

    def grad(self, A, a, parity=1.0):
        if self.iso:
            return sum(3 * wi * e[a] * self.nb(A, e, parity) for e, wi in zip(self.E, self.w) if e[a])
        return 0.5 * (self.nb(A, self.unit(a, 1), parity) - self.nb(A, self.unit(a, -1), parity))

    def step(self):
        d, p, phi = self.d, self.p, self.phi
        av = (self.T - p["Tc"]) / p["Tc"]
        psi = self.lap(phi)
        lam = self.lap(psi)
        mu = av * phi + p["b"] * phi ** 3 - p["kappa"] * psi + p["c"] * lam
        new = phi + p["Gamma"] * self.lap(mu)
        if self.hydro:
            gp = [self.grad(phi, a) for a in range(d)]
            gs = [self.grad(psi, a) for a in range(d)]
            iso = (av * phi ** 2 / 2 + 0.75 * p["b"] * phi ** 4
                   - p["kappa"] * (phi * psi + 0.5 * sum(g * g for g in gp))
                   + p["c"] * (phi * lam + 0.5 * psi * psi + sum(g * s for g, s in zip(gp, gs))))
            F = [torch.zeros_like(phi) for _ in range(d)]
            for a in range(d):
                for b in range(a, d):
                    P = p["kappa"] * gp[a] * gp[b] - p["c"] * (gp[a] * gs[b] + gp[b] * gs[a])
                    if a == b:
                        P = P + iso
                    par = -1.0 if (a == d - 1) != (b == d - 1) else 1.0
                    F[b] -= self.grad(P, a, par)
                    if a != b:
                        F[a] -= self.grad(P, b, par)
            del gp, gs, iso, lam, psi, mu
            n = sum(self.f)
            u = [(sum(e[a] * f for e, f in zip(self.E, self.f) if e[a]) + F[a] / 2) / n for a in range(d)]
            u2 = sum(v * v for v in u)
            uF = sum(v * g for v, g in zip(u, F))
            guo = 1 - 1 / (2 * self.tau)
            for i, (e, wi) in enumerate(zip(self.E, self.w)):
                eu = sum(c * v for c, v in zip(e, u) if c) if i else torch.zeros_like(n)
                eF = sum(c * g for c, g in zip(e, F) if c) if i else torch.zeros_like(n)
                feq = wi * n * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * u2)
                self.f[i] = self.f[i] - (self.f[i] - feq) / self.tau + guo * wi * (3 * (eF - uF) + 9 * eu * eF)
            post, out = self.f, []
            for i, e in enumerate(self.E):
                back = tuple(-c for c in e)
                s = self.nb(post[i], back)
                if self.walls and e[d - 1]:
                    opp = post[self.E.index(back)]
                    k = 0 if e[d - 1] > 0 else -1
                    s[:, k] = opp[:, k]
                out.append(s)
            self.f = out
            for a in range(d):
                new = new - self.grad(phi * u[a], a, -1.0 if a == d - 1 else 1.0)
        self.phi = new

    def heat(self):
        """Explicit sub-steps of the temperature, xi / n_sub each (a run takes no part beyond its own n_sub)."""
        ghost = 2 * self.T_w if self.t_mode == 1 else None
        ns = torch.tensor(self.nsub, device=self.T.device, dtype=torch.float64).view(self.xi.shape)
        for k in range(max(self.nsub)):
            T = self.T + torch.where(ns > k, self.xi / ns, 0.0) * self.lap(self.T, ghost)
            if self.walls and self.t_mode == 0:
                T[:, 0] = T[:, -1] = self.T_w
            self.T = T

    def heat_implicit(self):
        """(I - xi L) T' = T by Fourier modes along the periodic axes and a tridiagonal solve along the walls."""
        d, xi = self.d, float(self.xi.flatten()[0])
        L = self.T.shape[1]
        per = tuple(range(2, d + 1))
        X = torch.fft.fftn(self.T, dim=per)[0]
        c = [torch.cos(2 * math.pi * torch.arange(n, device=X.device, dtype=torch.float64) / n) for n in X.shape[1:]]
        cc = c[0] if d == 2 else c[0].view(-1, 1) + c[1].view(1, -1)
        off, diag = -xi, 1 + xi * (2 + 2 * (d - 1) - 2 * cc)
        j0, j1 = (1, L - 2) if self.t_mode == 0 else (0, L - 1)
        dg = [diag for _ in range(L)]
        rhs = [X[j].clone() for j in range(L)]
        if self.t_mode == 0:
            rhs[1] -= off * X[0]
            rhs[L - 2] -= off * X[L - 1]
        else:
            dg[0], dg[L - 1] = dg[0] - off, dg[L - 1] - off
            nper = math.prod(X.shape[1:])
            for j in (0, L - 1):
                rhs[j].view(-1)[0] += 2 * xi * self.T_w * nper
        cp = [None] * L
        for j in range(j0, j1 + 1):
            piv = dg[j] if j == j0 else dg[j] - off * cp[j - 1]
            cp[j] = off / piv
            rhs[j] = (rhs[j] if j == j0 else rhs[j] - off * rhs[j - 1]) / piv
        for j in range(j1 - 1, j0 - 1, -1):
            rhs[j] = rhs[j] - cp[j] * rhs[j + 1]
        self.T = torch.fft.ifftn(torch.stack(rhs)[None], dim=per).real

    def report(self):
        d, p, phi, N = self.d, self.p, self.phi, self.phi[0].numel()
        walls, iso = self.walls, self.iso
        self.iso = False                                   # the diagnostics are defined with the compact stencils
        g2 = [float((self.grad(phi, a) ** 2).sum()) for a in range(d)]
        links = sum((self.nb(phi, self.unit(a, 1)) - phi) ** 2 for a in range(d))
        av = (self.T - p["Tc"]) / p["Tc"]
        fe = (av * phi ** 2 / 2 + p["b"] * phi ** 4 / 4 + p["kappa"] * links / 2 + p["c"] * self.lap(phi) ** 2 / 2).sum()
        self.iso = iso
        lmin = min(phi.shape[1:])
        S = torch.fft.fftn(phi[0]).abs() ** 2 / N
        r2 = 0
        for a, n in enumerate(S.shape):
            i = torch.arange(n, device=S.device)
            k = torch.where(2 * i <= n, i, i - n).double() * lmin / n
            r2 = r2 + (k ** 2).view([-1 if b == a else 1 for b in range(d)])
        b = torch.floor(torch.sqrt(r2) + 0.5).long().flatten()
        B = lmin // 2
        ok = (b >= 1) & (b <= B)
        num = torch.zeros(B + 1, device=S.device, dtype=torch.float64).index_add_(0, b[ok], S.flatten()[ok])
        cnt = torch.zeros(B + 1, device=S.device, dtype=torch.float64).index_add_(0, b[ok], torch.ones_like(S.flatten()[ok]))
        Sb = num / cnt.clamp(min=1)
        top = Sb > 0.5 * Sb.max()
        kb = 2 * math.pi / lmin * torch.arange(B + 1, device=S.device)
        return {"mass": float(sum(f.sum() for f in self.f)), "free_energy": float(fe),
                "grad2": g2,
                "k_peak": float((kb * Sb)[top].sum() / Sb[top].sum()), "s_peak": float(Sb.max())}


def _noise(seed, n, amp):
    """The initial phi: SplitMix64 outputs k = 0 .. n - 1 of `seed`, the top 53 bits mapped to [-amp, amp)."""
    def shr(z, s):
        return (z >> s) & ((1 << (64 - s)) - 1)

    def i64(v):
        v &= (1 << 64) - 1
        return v - (1 << 64) if v >> 63 else v

    z = i64(seed) + (torch.arange(n, device="cuda", dtype=torch.int64) + 1) * i64(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * i64(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * i64(0x94D049BB133111EB)
    z = z ^ shr(z, 31)
    return amp * (2 * (shr(z, 11).double() * 2.0 ** -53) - 1)


def _start(shape, seeds, phys, walls, t_mode, T0, T_w, rnd):
    """phi and T of fresh lattices, as the state's precision holds them."""
    n = math.prod(shape)
    phi = torch.stack([rnd(_noise(s, n, phys["phi_amp"])).view(shape) for s in seeds])
    T = rnd(torch.full_like(phi, T0))
    if walls and t_mode == 0:
        T[:, 0] = T[:, -1] = rnd(torch.tensor(T_w, dtype=torch.float64, device="cuda"))
    return phi, T


def _f32(t):
    return t.float().double()


def _sur_net(params, x, dt=torch.float64):
    """The network in FP64 on normalised states x [B][NY][NX][4]; returns (y, parameters as leaves)."""
    leaves, off, v = [], 0, torch.from_numpy(params).cuda().to(dt)
    for cin, cout in SUR_LAYERS:
        leaves.append(v[off:off + 9 * cin * cout].view(9, cout, cin).clone().requires_grad_(True))
        off += 9 * cin * cout
        leaves.append(v[off:off + cout].clone().requires_grad_(True))
        off += cout

    def conv(h, W, b):
        hp = torch.cat([h[:, :, -1:], h, h[:, :, :1]], dim=2)
        hp = torch.nn.functional.pad(hp, (0, 0, 0, 0, 1, 1))
        NY, NX = h.shape[1:3]
        return b + sum(hp[:, t // 3:t // 3 + NY, t % 3:t % 3 + NX] @ W[t].T for t in range(9))

    h = torch.relu(conv(torch.nn.functional.pad(x, (0, 12)), leaves[0], leaves[1]))
    for l in range(1, 5):
        h = h + torch.relu(conv(h, leaves[2 * l], leaves[2 * l + 1]))
    return x + conv(h, leaves[10], leaves[11])[..., :4], leaves


def exact(case, seed):
    if case["kind"] == "lattice":
        kw = _kwargs(case, seed)
        phys = PHYSICS[case["physics"]]
        shape = (case["nz"], case["ny"], case["nx"])[3 - case["d"]:]
        rnd = _f32 if case["precision"] == "fp32" else (lambda t: t)
        phi, T = _start(shape, [seed], phys, case["walls"], case["t_mode"], kw["T0"], kw["T_w"], rnd)
        ex = _Exact(case["d"], case["walls"], case["t_mode"], case["stencil"], case["hydro"], phys, kw["T_w"], [case["xi"]],
                    [case["tau"]], phi, T)
        for _ in range(case["steps"]):
            ex.step()
            ex.heat_implicit() if case["solver"] == "implicit" else ex.heat()
        out = {"phi": ex.phi[0], "T": ex.T[0], "pop": torch.cat(ex.f)}
        if case["report"]:
            out["report"] = ex.report()
        return out
    if case["kind"] == "ensemble":
        members, out, phys = _ens_members(case, seed), {}, PHYSICS["config"]
        for i, n in enumerate(ENS_SIZES):
            ms = members[i::4]
            if ms:
                phi, T = _start((n, n), [m["seed"] for m in ms], phys, 1, 0, 1.1, case["tw"], _f32)
                ex = _Exact(2, 1, 0, case["stencil"], 1, phys, case["tw"], [m["xi"] for m in ms], [m["tau"] for m in ms], phi, T)
                for _ in range(case["steps"]):
                    ex.step()
                    ex.heat()
                out[f"n{n}"] = {"phi": ex.phi, "T": ex.T, "pop": torch.stack(ex.f, dim=1)}
        return out
    x, y = _sur_fields(case, seed)
    scale = torch.tensor(SUR_SCALE, device="cuda", dtype=torch.float64)
    offset = torch.tensor(SUR_OFFSET, device="cuda", dtype=torch.float64)
    nx = (x.double().permute(0, 2, 3, 1) - offset) / scale
    p0 = _sur_params(seed)
    if case["kind"] == "predict":
        with torch.no_grad():
            return {"y": (_sur_net(p0, nx)[0] * scale + offset).permute(0, 3, 1, 2)}
    sse, grads = 0.0, None                       # one state at a time: the batch's activations in FP64 are large
    for b in range(case["batch"]):
        yb, leaves = _sur_net(p0, nx[b:b + 1])
        loss = ((yb - (y[b:b + 1].double().permute(0, 2, 3, 1) - offset) / scale) ** 2).sum() / nx.numel()
        g = torch.autograd.grad(loss, leaves)
        sse += float(loss)
        grads = list(g) if grads is None else [u + v for u, v in zip(grads, g)]
    g = torch.cat([v.flatten() for v in grads])
    g = g * min(1.0, 1.0 / float(g.norm()))      # the global norm is clipped to 1
    m, v = 0.1 * g / (1 - 0.9), 0.001 * g * g / (1 - 0.999)
    step = case["lr"] * m / (v.sqrt() + 1e-8)
    return {"loss": sse, "params": (torch.from_numpy(p0).cuda().double() - step).cpu().numpy()}
