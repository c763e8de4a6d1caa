"""Timing cases of the TILD framework: what a user's program has it do,
through the public entry points of the binding, over the sizes in use.

A case is one system (chains, box, grid, precision, options) and one kind of
call:

  steps       t.step(k), then the positions and velocities are read
  observe     energies, forces and the density of the current state
  gradient    the pieces of one differentiable loss: energy gradient, force
              vector-Jacobian product, density vector-Jacobian product
  trajectory  reverse-mode derivatives through a window of steps
  batch       many uneven replicas stepped together, then read

Positions are returned as displacements from the start of the case (minimum
image), as a program that accumulates mean-square displacements takes them.
"""
import math

import numpy as np
import torch

from paper_2302_02474_gb300 import binding as B
from paper_2302_02474_gb300.trajectory import trajectory_vjp

# Grid edges of the tiled kernels; every other edge runs on the any-size ones.
TILED = (16, 24, 32, 40, 48, 64, 80, 128)

_BASE = dict(kind="steps", dim=3, mix="diblock", species=2, order=1, precision="fp32", scheme="gjf", method="ik",
             charged=False, a=0.5, chi=1.0, kappa=25.0, dt=0.005, steps=20, every=20, replicas=1)


def _case(**kw):
    c = dict(_BASE)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest replica of a parameter scan, sampled often: launches and latency
        _case(name="melt_4k_24", chains=203, N=20, n_a=10, L=14.4, n=24, steps=20),
        # the plain FP64 validation system (20,000 beads, 32^3, 100 steps)
        _case(name="melt_20k_32_fp64", chains=1000, N=20, n_a=10, L=20.0, n=32, kappa=20.0, precision="fp64", steps=100),
        # the two-dimensional setting of the method's input listing: a 65 x 65 grid
        _case(name="listing_2d_65", dim=2, chains=250, N=20, n_a=10, L=32.5, n=65, chi=1.4375 * 5000 / 32.5**2,
              kappa=1.5625 * 5000 / 32.5**2, steps=40),
        # charged chains (35,588 beads of a coacervate), third-order weights, velocity-Verlet
        _case(name="coacervate_36k_48", chains=434, N=82, n_a=41, L=26.0, n=48, order=3, scheme="vv", charged=True, steps=40),
        # three species on an odd grid
        _case(name="ternary_55k_45", mix="block", species=3, chains=1851, N=30, n_a=10, L=25.2, n=45, steps=20),
        # energy-conserving (analytic) forces with second-order weights
        _case(name="analytic_400k_80", chains=20011, N=20, n_a=7, L=40.0, n=80, order=2, method="analytic", steps=40),
        # the production melt: 1.6M beads on 128^3
        _case(name="melt_1p6M_128", chains=80000, N=20, n_a=8, L=64.0, n=128, chi=0.8, steps=40),
        # the largest: ternary blend with a compatibiliser, 6.4M beads on 256^3
        _case(name="blend_6p4M_256", mix="blend", chains=80000, N=32, n_a=16, L=128.0, n=256, a=0.6, chi=0.5, kappa=30.0,
              steps=20),
        # one sample of the production melt's observables
        _case(name="observe_1p6M_128", kind="observe", chains=80000, N=20, n_a=8, L=64.0, n=128, chi=0.8),
        # derivatives of one differentiable loss on the 200k-bead melt
        _case(name="gradient_200k_64", kind="gradient", chains=10000, N=20, n_a=10, L=32.0, n=64),
        # reverse mode through a checkpointed window of the same melt; second-order
        # weights, whose derivatives are continuous across cells
        _case(name="trajectory_200k_64", kind="trajectory", chains=10000, N=20, n_a=10, L=32.0, n=64, order=2, steps=20, every=10),
        # a parameter scan: uneven replicas on 24^3 to 64^3
        _case(name="batch_64", kind="batch", chains=1100, N=20, n_a=10, L=24.0, n=64, steps=60, replicas=64),
    ]


def _loguniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "steps", "observe", "gradient", "trajectory", "batch"])
    N = rng.choice([4, 8, 13, 20, 20, 32, 50, 82])
    frac = rng.choice([0.25, 0.4, 0.5])
    c = _case(kind=kind, N=N, n_a=max(1, int(N * frac)), a=round(rng.uniform(0.4, 0.7), 3), chi=round(rng.uniform(0.2, 1.5), 3),
              kappa=round(rng.uniform(20.0, 30.0), 2))
    if kind == "batch":
        c.update(N=20, n_a=10, replicas=rng.randrange(8, 65), n=64, L=24.0, chains=rng.randrange(200, 1400),
                 steps=rng.choice([20, 40, 60]))
        return c
    if kind == "steps" and rng.random() < 0.12:
        n = rng.randrange(33, 130)
        L = round(n * rng.uniform(0.45, 0.6), 3)
        beads = int(_loguniform(rng, 1.5, 6.0) * n * n)
        rho0 = beads / L**2
        c.update(dim=2, n=n, L=L, chains=max(1, beads // N), chi=round(rng.uniform(0.5, 1.4375) * rho0, 4),
                 kappa=round(1.5625 * rho0, 4), order=rng.choice([1, 1, 2, 3]), steps=rng.choice([20, 40]))
        return c
    if kind == "steps" and rng.random() < 0.2:
        n = rng.randrange(15, 66)  # mostly sizes of the any-size kernels
    elif kind in ("gradient", "trajectory"):
        n = rng.choice([24, 32, 40, 48, 64, 64])
    else:
        n = rng.choice(TILED[1:] if kind == "steps" else (32, 48, 64, 80, 128))
    L = round(n * rng.uniform(0.5, 0.67), 3)
    beads = int(_loguniform(rng, 0.2, 1.0) * n**3)
    c.update(n=n, L=L, chains=max(1, beads // N), order=rng.choice([1, 1, 1, 1, 2, 3, 4]))
    if kind == "trajectory":
        c.update(steps=rng.choice([5, 10, 20]), every=rng.choice([5, 10]), order=rng.choice([2, 2, 3]), scheme=rng.choice(["gjf", "gjf", "vv"]))
        return c
    if kind == "steps":
        c.update(steps=rng.choice([10, 20, 40]), scheme=rng.choice(["gjf", "gjf", "gjf", "vv", "em"]))
    if n <= 64 and rng.random() < 0.2:
        c.update(precision="fp64")
    if kind != "gradient" and n in TILED:
        option = rng.choice(["", "", "", "analytic", "charged", "blend", "species"])
        if option == "analytic":
            c.update(method="analytic", order=max(2, c["order"]))  # first-order weights: a force with jumps
        elif option == "charged":
            c.update(charged=True)
        elif option == "blend":
            c.update(mix="blend", chains=max(2, c["chains"] * 2 // 5))
        elif option == "species":
            c.update(mix="block", species=rng.choice([3, 4]), N=20, chains=max(1, beads // 20))
    return c


# ------------------------------------------------------------------ systems

_CHARGES = (1.0, -1.0, 1.0, 0.5)  # q_A, q_B, Bjerrum length, charge spreading length


def _moltypes(c):
    """(chains, N, n_a) per molecule type."""
    if c["mix"] == "blend":
        return [(c["chains"], c["N"], c["N"]), (c["chains"], c["N"], 0), (max(1, c["chains"] // 2), c["N"], c["N"] // 2)]
    return [(c["chains"], c["N"], c["n_a"])]


def _replicas(c):
    """The systems of a case: itself, or the uneven replicas of a batch
    (4,000 to 40,000 beads around its mean, boxes of 16 to 32, spacings near 0.5 to 0.67)."""
    if c["kind"] != "batch":
        return [c]
    rng = np.random.Generator(np.random.PCG64(c["chains"]))
    sizes = np.array([24, 32, 40, 48, 64])
    out = []
    for _ in range(c["replicas"]):
        L = float(rng.uniform(16.0, 32.0))
        n = int(sizes[np.argmin(np.abs(sizes - L / rng.uniform(0.5, 0.67)))])
        chains = int(min(2000, max(200, c["chains"] * rng.uniform(0.2, 1.8))))
        out.append(dict(c, chains=chains, L=L, n=n, chi=float(rng.uniform(0.2, 1.5))))
    return out


def _beads(c):
    return sum(k * N for k, N, _ in _moltypes(c))


def _species(c, device):
    if c["mix"] == "block":
        one = torch.arange(c["N"], device=device) * c["species"] // c["N"]
        return one.repeat(c["chains"])
    return torch.cat([(torch.arange(N, device=device) >= n_a).long().repeat(k) for k, N, n_a in _moltypes(c)])


def _chi_matrix(c):
    S = c["species"]
    return [[0.0 if i == j else c["chi"] * (1.0 + 0.25 * (i + j)) for j in range(S)] for i in range(S)]


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _dtype(c):
    return torch.float64 if c["precision"] == "fp64" else torch.float32


def _inputs(c, seed):
    """Random-walk chains and Maxwell-Boltzmann velocities, (beads, 3) each,
    in the context's precision."""
    dev, D = _device(), c["dim"]
    g = torch.Generator(device=dev).manual_seed(int(seed) * 1009 + 17)
    parts = []
    for k, N, _ in _moltypes(c):
        first = torch.rand(k, 1, D, generator=g, device=dev, dtype=torch.float64) * c["L"]
        u = torch.randn(k, N - 1, D, generator=g, device=dev, dtype=torch.float64)
        u = u / u.norm(dim=2, keepdim=True)
        parts.append(torch.cat([first, first + u.cumsum(1)], 1).reshape(-1, D))
    r = torch.remainder(torch.cat(parts), c["L"]).to(_dtype(c))
    r = torch.where(r >= c["L"], torch.zeros_like(r), r)
    v = torch.randn(r.shape, generator=g, device=dev, dtype=torch.float64).to(_dtype(c))
    if D == 2:
        r, v = (torch.cat([x, torch.zeros_like(x[:, :1])], 1) for x in (r, v))
    return r.contiguous(), v.contiguous()


def _adjoints(c, seed):
    """The adjoints that reach the library from the rest of a loss."""
    dev = _device()
    g = torch.Generator(device=dev).manual_seed(int(seed) * 2003 + 5)
    lam = torch.randn(_beads(c), 3, generator=g, device=dev, dtype=torch.float64).to(_dtype(c))
    vbar = torch.randn(_beads(c), 3, generator=g, device=dev, dtype=torch.float64).to(_dtype(c))
    psi = None
    if c["kind"] == "gradient":
        psi = torch.randn(c["species"], c["n"], c["n"], c["n"], generator=g, device=dev, dtype=torch.float64).to(_dtype(c))
    return lam, vbar, psi


def _context(c, seed, r, v):
    t = B.Tild(c["L"], c["n"], c["order"], c["precision"], 777 + int(seed), dim=c["dim"])
    t.set_chains(_moltypes(c), 1.0)
    if c["species"] > 2:
        t.set_species(c["species"], _species(c, "cpu").numpy())
    t.set_interactions(c["chi"], c["kappa"], c["a"])
    if c["species"] > 2:
        t.set_chi_matrix(_chi_matrix(c))
    t.set_integrator(c["dt"], 1.0, 1.0, 1.0)
    if c["charged"]:
        t.set_electrostatics(*_CHARGES)
    if c["method"] != "ik":
        t.set_force_method(c["method"])
    if c["scheme"] != "gjf":
        t.set_scheme(c["scheme"])
    t.set_positions(r)
    t.set_velocities(v)
    return t


def prepare(case, seed):
    c = dict(_BASE, **case)
    reps = _replicas(c)
    rs, vs = zip(*[_inputs(q, seed * 4099 + k) for k, q in enumerate(reps)])
    torch.cuda.synchronize()  # the contexts read the inputs on their own streams
    ts = [_context(q, seed * 4099 + k, r, v) for k, (q, r, v) in enumerate(zip(reps, rs, vs))]
    r0 = torch.cat(rs)
    s = dict(case=c, t=ts[0], ts=ts, r0=r0, r=torch.empty_like(r0), v=torch.empty_like(r0))
    if c["kind"] == "batch":
        counts = [len(r) for r in rs]
        s["batch"] = B.TildBatch(ts)
        s["L"] = torch.cat([torch.full((k, 1), q["L"], dtype=r0.dtype, device=r0.device) for k, q in zip(counts, reps)])
        s["rs"], s["vs"] = s["r"].split(counts), s["v"].split(counts)
    else:
        s["L"] = c["L"]
    if c["kind"] in ("gradient", "trajectory"):
        s["lam"], s["vbar"], s["psi"] = _adjoints(c, seed)
    if c["kind"] == "gradient":
        s["dU"], s["jt"], s["dens"] = (torch.empty_like(r0) for _ in range(3))
    if c["kind"] == "observe":
        s["f"] = torch.empty_like(r0)
        s["rho"] = torch.empty(c["species"], c["n"], c["n"], c["n"], dtype=r0.dtype, device=r0.device)
    torch.cuda.synchronize()
    return s


def _displacement(s):
    d = s["r"] - s["r0"]
    return d - s["L"] * torch.round(d / s["L"])


def run(s):
    c, t = s["case"], s["t"]
    if c["kind"] == "steps":
        t.step(c["steps"])
        t.positions(out=s["r"])
        t.velocities(out=s["v"])
        return {"dr": _displacement(s), "v": s["v"]}
    if c["kind"] == "batch":
        s["batch"].step(c["steps"])
        s["batch"].synchronize()
        for q, r, v in zip(s["ts"], s["rs"], s["vs"]):
            q.positions(out=r)
            q.velocities(out=v)
        return {"dr": _displacement(s), "v": s["v"]}
    if c["kind"] == "observe":
        _, e = t.compute(out=s["f"])
        t.density(out=s["rho"])
        return {"forces": s["f"], "rho": s["rho"], "bond": e["bond"], "chi": e["chi"], "kappa": e["kappa"],
                "elec": e["elec"], "kinetic": e["kinetic"]}
    if c["kind"] == "gradient":
        e, _ = t.energy_gradient(out=s["dU"])
        _, th = t.force_vjp(s["lam"], out=s["jt"])
        t.density_vjp(s["psi"], out=s["dens"])
        return {"dU_dr": s["dU"], "energy": e["energy"], "dU_dchi": e["dU_dchi"], "dU_dkappa": e["dU_dkappa"],
                "dU_da": e["dU_da"], "jt": s["jt"], "jt_theta": [th["chi"], th["kappa"], th["a"]], "dens": s["dens"]}
    g = trajectory_vjp(t, c["steps"], s["lam"], s["vbar"], c["every"])
    dt = s["r0"].dtype
    return {"r0": g["r0"].to(dt), "v0": g["v0"].to(dt), "theta": [g["chi"], g["kappa"], g["a"]]}


# --------------------------------------------------------------------- work


def _work_one(c):
    w = 8.0 if c["precision"] == "fp64" else 4.0
    N, D, S = _beads(c), c["dim"], c["species"]
    M = float(c["n"]) ** D
    F = 1 if c["method"] == "analytic" else D  # fields per species at the beads
    P3 = float((c["order"] + 1) ** D)
    fft = 2.5 * M * math.log2(M)  # one real field
    # a step: bead state read and written; density written and read, force fields written and read
    step = {"bytes": 4 * D * w * N + 2 * S * w * M * (1 + F), "flops": N * (P3 * (2 * F + 4) + 150) + S * (1 + F) * fft}
    # a force VJP: positions and adjoints in, result out; the spread adjoint (D fields) and psi (1 field)
    vjp = {"bytes": 3 * D * w * N + 2 * S * w * M * (D + 1), "flops": N * P3 * (4 * D + 8 * D) + S * (D + 1) * fft}
    return step, vjp, {"bytes": 2 * D * w * N, "flops": 0.0}


def work(case):
    c = dict(_BASE, **case)
    total = {"bytes": 0.0, "flops": 0.0}
    for q in _replicas(c):
        step, vjp, read = _work_one(q)
        parts = {"steps": [(step, c["steps"]), (read, 1)], "batch": [(step, c["steps"]), (read, 1)], "observe": [(step, 1)],
                 "gradient": [(step, 1), (vjp, 1), (read, 2)], "trajectory": [(step, c["steps"]), (vjp, c["steps"]), (read, 2)]}
        for p, k in parts[c["kind"]]:
            for key in total:
                total[key] += k * p[key]
    return total


# -------------------------------------------------------------------- exact
# The method in 64 bits with plain torch: B-spline weights, torch.fft, the
# integrators' textbook forms, derivatives from torch.autograd.


def _bspline(s, P):
    """First grid point, weights and their derivatives in s ([N] -> [N, P])."""
    shift = 0.5 * (P % 2)
    cell = torch.floor(s.detach() + shift)
    u = s + shift - cell
    w, prev = [1.0 - u, u], [torch.ones_like(u)]
    for k in range(3, P + 1):
        at = lambda i: w[i] if 0 <= i < len(w) else 0.0  # noqa: E731
        prev, w = w, [((u + k - 1 - j) * at(j - 1) + (1 + j - u) * at(j)) / (k - 1) for j in range(k)]
    at = lambda i: prev[i] if 0 <= i < len(prev) else 0.0  # noqa: E731
    dw = [at(j - 1) - at(j) + torch.zeros_like(u) for j in range(P)]
    j0 = cell.long() - (P // 2 - 1 if P % 2 == 0 else (P - 1) // 2)
    return j0, torch.stack(w, -1), torch.stack(dw, -1)


class _Exact:
    def __init__(self, c, seed):
        self.c, self.seed = c, 777 + int(seed)
        self.dev = dev = _device()
        self.D, self.n, self.L, self.P = c["dim"], c["n"], c["L"], c["order"] + 1
        self.M, self.N = self.n**self.D, _beads(c)
        self.V = self.L**self.D
        self.dV, self.rho0 = self.V / self.M, self.N / self.V
        self.S = c["species"]
        self.sp = _species(c, dev)
        chi = _chi_matrix(c) if self.S > 2 else [[0.0, c["chi"]], [c["chi"], 0.0]]
        self.X = torch.tensor(chi, dtype=torch.float64, device=dev)
        f = torch.fft.fftfreq(self.n, 1.0 / self.n, dtype=torch.float64, device=dev) * (2 * math.pi / self.L)
        g = f.clone()
        if self.n % 2 == 0:
            g[self.n // 2] = 0.0
        shape = lambda d: [self.n if e == self.D - 1 - d else 1 for e in range(self.D)]  # noqa: E731  (x fastest)
        self.k2 = sum((f**2).view(shape(d)) for d in range(self.D))
        self.kg = [g.view(shape(d)) for d in range(self.D)]
        starts, i = [], 0
        for k, N, _ in _moltypes(c):
            starts.append((i, k, N))
            i += k * N
        self.bonds = torch.cat([(i + torch.arange(k, device=dev)[:, None] * N + torch.arange(N - 1, device=dev)).reshape(-1)
                                for i, k, N in starts])
        self.ids = torch.arange(self.N, device=dev)

    def stencil(self, r):
        """Grid indices [N, P^D], weights, and the weights' gradients per axis."""
        ax = [_bspline(r[:, d] * (self.n / self.L), self.P) for d in range(self.D)]
        idx, w, dw = None, None, [None] * self.D
        for d in range(self.D):
            j = torch.remainder(ax[d][0][:, None] + torch.arange(self.P, device=self.dev), self.n) * self.n**d
            if idx is None:
                idx, w, dw[0] = j, ax[d][1], ax[d][2]
                continue
            mix = lambda p, q: (p[:, :, None] * q[:, None, :]).reshape(len(r), -1)  # noqa: E731
            idx = (idx[:, :, None] + j[:, None, :]).reshape(len(r), -1)
            dw = [mix(x, ax[d][1]) if x is not None else None for x in dw]
            dw[d] = mix(w, ax[d][2])
            w = mix(w, ax[d][1])
        return idx, w, [x * (self.n / self.L) for x in dw]

    def density(self, idx, w):
        flat = (self.sp[:, None] * self.M + idx).reshape(-1)
        rho = torch.zeros(self.S * self.M, dtype=torch.float64, device=self.dev).index_add(0, flat, w.reshape(-1) / self.dV)
        return rho.view([self.S] + [self.n] * self.D)

    def potentials(self, rho, theta):
        """Spectra of the species' potentials."""
        chi, kappa, a = theta
        X = self.X if self.S > 2 else torch.stack([torch.stack([0 * chi, chi]), torch.stack([chi, 0 * chi])])
        z = torch.fft.fftn(rho, dim=list(range(1, self.D + 1)))
        w = torch.exp(-self.k2 * a**2) * torch.einsum("kl,l...->k...", ((X + kappa) / self.rho0).to(z.dtype), z)
        if self.c["charged"]:
            q = torch.tensor(_CHARGES[:2], dtype=torch.float64, device=self.dev)
            w = w + torch.einsum("k,...->k...", q.to(z.dtype), self.coulomb() * torch.einsum("k,k...->...", q.to(z.dtype), z))
        return z, w

    def coulomb(self):
        k2 = torch.where(self.k2 == 0, torch.ones_like(self.k2), self.k2)
        return torch.where(self.k2 == 0, 0.0, 4 * math.pi * _CHARGES[2] * torch.exp(-self.k2 * _CHARGES[3] ** 2) / k2)

    def theta(self):
        return [torch.tensor(float(self.c[k]), dtype=torch.float64, device=self.dev) for k in ("chi", "kappa", "a")]

    def bond_vectors(self, r):
        d = r[self.bonds + 1, : self.D] - r[self.bonds, : self.D]
        return d - self.L * torch.round(d.detach() / self.L)

    def forces(self, r, theta):
        r = r[:, : self.D]
        idx, w, dw = self.stencil(r)
        _, wk = self.potentials(self.density(idx, w), theta)
        dims = list(range(1, self.D + 1))
        own = (self.sp[:, None] * self.M + idx).reshape(-1)
        read = lambda field: field.reshape(-1)[own].view(idx.shape)  # noqa: E731
        if self.c["method"] == "analytic":
            pot = read(torch.fft.ifftn(wk, dim=dims).real)
            f = torch.stack([-(x * pot).sum(1) for x in dw], 1)
        else:
            f = torch.stack([-(w * read(torch.fft.ifftn(1j * self.kg[d] * wk, dim=dims).real)).sum(1) for d in range(self.D)], 1)
        b = 3.0 * self.bond_vectors(r)
        return f.index_add(0, self.bonds, b).index_add(0, self.bonds + 1, -b)

    def energies(self, r, theta):
        chi, kappa, a = theta
        r = r[:, : self.D]
        idx, w, _ = self.stencil(r)
        z = torch.fft.fftn(self.density(idx, w), dim=list(range(1, self.D + 1)))
        u = torch.exp(-self.k2 * a**2)
        f = self.dV**2 / self.V
        pair = lambda i, j: (u * (z[i].conj() * z[j]).real).sum()  # noqa: E731
        e = {"bond": 1.5 * (self.bond_vectors(r) ** 2).sum()}
        if self.S > 2:
            e["chi"] = f / self.rho0 * sum(self.X[i, j] * pair(i, j) for i in range(self.S) for j in range(i + 1, self.S))
        else:
            e["chi"] = f / self.rho0 * chi * pair(0, 1)
        tot = u * z.sum(0).abs() ** 2
        e["kappa"] = f * kappa / (2 * self.rho0) * (tot.sum() - tot.reshape(-1)[0])
        e["elec"] = torch.zeros((), dtype=torch.float64)
        if self.c["charged"]:
            e["elec"] = f / 2 * (self.coulomb() * (_CHARGES[0] * z[0] + _CHARGES[1] * z[1]).abs() ** 2).sum()
        return e

    def noise(self, step):
        """Three normals per bead: Philox4x32-10, counter (id, step, 0, 0), key = seed."""
        m32 = 0xFFFFFFFF
        c = [self.ids.clone(), torch.full_like(self.ids, step & m32), torch.full_like(self.ids, (step >> 32) & m32),
             torch.zeros_like(self.ids)]
        k0, k1 = self.seed & m32, (self.seed >> 32) & m32
        for _ in range(10):
            p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
            c = [((p1 >> 32) & m32) ^ c[1] ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ c[3] ^ k1, p0 & m32]
            k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
        u = [(x.double() + 0.5) / 2.0**32 for x in c]
        m1, m2 = torch.sqrt(-2 * torch.log(u[0])), torch.sqrt(-2 * torch.log(u[2]))
        two_pi = 2 * math.pi
        return torch.stack([m1 * torch.cos(two_pi * u[1]), m1 * torch.sin(two_pi * u[1]), m2 * torch.cos(two_pi * u[3])], 1)[:, : self.D]

    def trajectory(self, r, v, K, theta):
        """Positions (not wrapped) and velocities after K steps."""
        dt = self.c["dt"]
        r, v = r[:, : self.D], v[:, : self.D]
        f = self.forces(r, theta)
        if self.c["scheme"] == "em":
            for s in range(K):
                r = r + dt * f + math.sqrt(2 * dt) * self.noise(s + 1)
                f = self.forces(r, theta)
            return r, torch.zeros_like(v)
        if self.c["scheme"] == "vv":
            h, sig = dt / 2, math.sqrt(2 / dt)
            u = (v - h * (f + sig * self.noise(0))) / (1 - h)
            for s in range(K):
                u = u + dt * (f - u + sig * self.noise(s))
                r = r + dt * u
                f = self.forces(r, theta)
            return r, u + h * (f - u + sig * self.noise(K))
        b, a = 1 / (1 + dt / 2), (1 - dt / 2) / (1 + dt / 2)
        for s in range(K):
            beta = math.sqrt(2 * dt) * self.noise(s + 1)
            r = r + b * dt * (v + dt / 2 * f + beta / 2)
            f1 = self.forces(r, theta)
            v = a * v + dt / 2 * (a * f + f1) + b * beta
            f = f1
        return r, v


def _three(x):
    return x if x.shape[1] == 3 else torch.cat([x, torch.zeros_like(x[:, :1])], 1)


def exact(case, seed):
    c = dict(_BASE, **case)
    if c["kind"] in ("steps", "batch"):
        drs, vs = [], []
        for k, q in enumerate(_replicas(c)):
            r, v = (x.double() for x in _inputs(q, seed * 4099 + k))
            m = _Exact(q, seed * 4099 + k)
            r1, v1 = m.trajectory(r, v, c["steps"], m.theta())
            d = r1 - r[:, : c["dim"]]
            drs.append(_three(d - q["L"] * torch.round(d / q["L"])))
            vs.append(_three(v1))
        return {"dr": torch.cat(drs), "v": torch.cat(vs)}
    s0 = seed * 4099
    r, v = (x.double() for x in _inputs(c, s0))
    m = _Exact(c, s0)
    if c["kind"] == "observe":
        e = m.energies(r, m.theta())
        f = m.forces(r, m.theta())
        idx, w, _ = m.stencil(r)
        return {"forces": f, "rho": m.density(idx, w), "bond": float(e["bond"]), "chi": float(e["chi"]),
                "kappa": float(e["kappa"]), "elec": float(e["elec"]), "kinetic": float(0.5 * (v**2).sum())}
    lam, vbar, psi = (None if x is None else x.double() for x in _adjoints(c, seed))
    r.requires_grad_()
    theta = [x.requires_grad_() for x in m.theta()]
    if c["kind"] == "gradient":
        e = m.energies(r, theta)
        U = e["bond"] + e["chi"] + e["kappa"] + e["elec"]
        dU = torch.autograd.grad(U, [r] + theta)
        jt = torch.autograd.grad((m.forces(r, theta) * lam).sum(), [r] + theta)
        idx, w, _ = m.stencil(r)
        dens = torch.autograd.grad((m.density(idx, w) * psi).sum(), r)[0]
        return {"dU_dr": dU[0], "energy": float(U), "dU_dchi": float(dU[1]), "dU_dkappa": float(dU[2]), "dU_da": float(dU[3]),
                "jt": jt[0], "jt_theta": [float(x) for x in jt[1:]], "dens": dens}
    v.requires_grad_()
    rK, vK = m.trajectory(r, v, c["steps"], theta)
    g = torch.autograd.grad((rK * lam).sum() + (vK * vbar).sum(), [r, v] + theta)
    return {"r0": g[0], "v0": g[1], "theta": [float(x) for x in g[2:]]}
