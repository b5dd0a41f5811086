"""Performance cases of the MXE hot path: what a program that uses this
package has it do, through `MxeSystem`, `MxeBatch` and `free_energy`.

Kinds (`case["kind"]`):
  evaluate   new positions, widths and fractions in; lists built; free energy
             and every gradient out (the call of a driver that moves the sites
             itself, and of every monitoring point of a run)
  step       one step of the staggered scheme of the paper (Sec. 4) from given
             inputs: lists, free energy and excess chemical potentials, one
             Euler step of the master equation, `iters` FIRE iterations
  diffuse    lists, free energy and gradients, one Euler step, no relaxation
             (diffusion on an interstitial sublattice)
  run        `steps` staggered steps of a batch of independent systems as one
             graph launch (an ensemble over temperatures and vacancy contents)
  gradient   forward and backward of the differentiable free energy
  hvp        Hessian-vector product and term sensitivities (the inner call of
             every derivative of a relaxed state)

Precisions are the library's three: "fp64" (the default of `MxeSystem`),
"mixed" and "ff".  The two FP32 modes form forces, and with them relaxed
positions and widths, from FP32 node arithmetic, so a program that asked for
them keeps those as float32; chemical potentials, energies and molar fractions
are accurate to FP64 budgets in every mode and stay float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1910_01235_gb300 import mxe as M
from paper_1910_01235_gb300 import workloads as W

KB = 8.617333262e-5
SQRT6 = math.sqrt(6.0)
DEV = "cuda:0" if torch.cuda.is_available() else "cpu"


def listed():
    return [
        # the smallest call: a 500-site vacancy lattice evaluated once per move of an outer program
        dict(name="evaluate_500_ff", kind="evaluate", system="vacancy", cells=5, precision="ff"),
        # interactive runs on a small cell at the library's default precision
        dict(name="step_500_fp64", kind="step", system="vacancy", cells=5, precision="fp64", iters=10),
        # equilibration of a small alloy cell with a stable potential: many cheap iterations
        dict(name="step_2k_mixed", kind="step", system="alloy_stable", cells=8, precision="mixed", iters=40),
        # production step of a mid-sized alloy at the default precision, odd number of cells
        dict(name="step_20k_fp64", kind="step", system="alloy", cells=17, precision="fp64", iters=10),
        # the same step with FP64 sums of FP32 node arithmetic
        dict(name="step_55k_mixed", kind="step", system="alloy", cells=24, precision="mixed", iters=10),
        # the benchmark's step: 256,000-site binary alloy, float-float sums
        dict(name="step_256k_ff", kind="step", system="alloy", cells=40, precision="ff", iters=10),
        # the paper's scaling shape: copper with one vacancy, monitored free energy and gradients
        dict(name="evaluate_864k_ff", kind="evaluate", system="copper", cells=60, precision="ff"),
        # hydrogen-like solute on the octahedral sublattice of a 4-million-site slab
        dict(name="diffuse_4m_ff", kind="diffuse", system="slab", cells=100, precision="ff"),
        # ensemble of small lattices over temperature and vacancy content
        dict(name="run_512_systems_ff", kind="run", system="ensemble", count=512, cmax=16, steps=2, precision="ff",
             iters=10),
        # free energy of a surface alloy as a differentiable scalar inside an autograd program
        dict(name="gradient_108k_fp64", kind="gradient", system="surface", cells=30, precision="fp64"),
        # one Hessian-vector product of the implicit-function derivative of a relaxed alloy
        dict(name="hvp_11k_fp64", kind="hvp", system="alloy_stable", cells=14, precision="fp64"),
        # the exact (non-Taylor) embedding average where the Taylor form is checked against it
        dict(name="evaluate_5k_exact_fp64", kind="evaluate", system="alloy", cells=11, precision="fp64",
             embedding="exact"),
    ]


def _cells(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["evaluate", "step", "step", "diffuse", "run", "gradient", "hvp"])
    precision = rng.choice(["fp64", "mixed", "ff"])
    fp64 = precision == "fp64"
    if kind == "evaluate":
        if rng.random() < 0.25:
            return dict(kind=kind, system=rng.choice(["alloy", "vacancy"]), cells=_cells(rng, 4, 14), precision="fp64",
                        embedding="exact")
        return dict(kind=kind, system=rng.choice(["vacancy", "alloy", "copper", "surface"]),
                    cells=_cells(rng, 5, 34 if fp64 else 58), precision=precision)
    if kind == "step":
        return dict(kind=kind, system=rng.choice(["vacancy", "alloy", "alloy_stable"]),
                    cells=_cells(rng, 5, 19 if fp64 else 40), precision=precision, iters=rng.choice([6, 8, 10]))
    if kind == "diffuse":
        return dict(kind=kind, system="slab", cells=_cells(rng, 8, 30 if fp64 else 80), precision=precision)
    if kind == "run":
        return dict(kind=kind, system="ensemble", count=_cells(rng, 3, 40 if fp64 else 400), cmax=rng.randint(4, 11),
                    steps=rng.choice([1, 2, 3]), precision=precision, iters=rng.choice([5, 8, 10]))
    if kind == "gradient":
        return dict(kind=kind, system=rng.choice(["surface", "alloy", "vacancy"]), cells=_cells(rng, 5, 28),
                    precision="fp64")
    return dict(kind=kind, system=rng.choice(["vacancy_stable", "alloy_stable"]), cells=_cells(rng, 4, 16),
                precision="fp64")


# ------------------------------------------------------------------ inputs
def _host_systems(case, seed):
    """The host-side systems of a case: lattice recipes of the package, sites
    displaced by up to 0.05 A per axis and widths by up to 0.02 A (a thermal
    state; the relaxations start from it).  Ensembles start from the lattice
    with drawn temperatures and vacancy fractions, the slab with drawn solute
    fractions."""
    name, cells = case["system"], case.get("cells", 0)
    if name == "ensemble":
        # sizes of the recipe's own seed (the layout belongs to the case), states of the given one
        systems = W.config_ensemble(case["count"], 4, case["cmax"], pot=W.potential_variant_s())
        rng = np.random.default_rng(seed)
        for s in systems:
            s.T = np.full(s.n, rng.uniform(300.0, 1200.0))
            s.x = 1.0 - (1.0 - s.x) * rng.uniform(0.5, 1.5, s.x.shape)
        return systems
    if name == "vacancy":
        s = W.config_vacancy_lattice(cells)
    elif name == "vacancy_stable":
        s = W.config_vacancy_lattice(cells, pot=W.potential_variant_s())
    elif name == "copper":
        s = W.config_cu_vacancy(cells)
    elif name == "surface":
        s = W.config_surface_alloy(cells, seed=seed)
    elif name == "slab":
        return [W.config_interstitial_slab(cells, cells, max(4, cells // 2), seed=seed)]
    else:
        s = W.config_binary_alloy(cells, seed=seed)
        if name == "alloy_stable":
            s.pot = W.potential_binary_variant_s()
    return [W.perturb(s, 0.05, 0.02, seed=seed + 1)]


def _dt(case, s):
    """Euler step: the recipe's own; a hundredth of it in the lattices whose
    vacancy is a whole empty site (its rates are far above the mean) and a
    millionth in the slab (the solute's chemical potentials differ by electron
    volts between the free surface and the sites below it)."""
    return s.dt_default() * {"vacancy": 0.01, "copper": 0.01, "vacancy_stable": 0.01, "slab": 1e-6}.get(case["system"], 1.0)


def prepare(case, seed):
    systems = _host_systems(case, seed)
    if case["kind"] == "run":
        g = M.MxeBatch(systems, case["precision"], device=DEV)
        g.set_dt_scale([s.dt_default() for s in systems])
    else:
        g = M.MxeSystem(systems[0], case["precision"], device=DEV)
    if case.get("embedding"):
        g.set_embedding(case["embedding"])
    g.build_neighbors()
    st = dict(case=case, g=g, q=g.q.clone(), sigma=g.sigma.clone(), x=g.x.clone(), dt=_dt(case, systems[0]),
              fire=M.make_fire(check_every=case.get("iters", 0) + 1))
    if case["kind"] == "hvp":
        st["tangent"] = tuple(torch.as_tensor(t, device=DEV) for t in _tangent(systems[0], seed))
    return st


def _tangent(s, seed):
    rng = np.random.default_rng(seed + 2)
    return rng.normal(0.0, 1.0, (3, s.n)), rng.normal(0.0, 1.0, s.n), rng.normal(0.0, 0.1, (s.S, s.n))


# ------------------------------------------------------------------ one pass
def _kept(case, t):
    """Forces, relaxed positions and widths as a program of this precision keeps them."""
    return t if case["precision"] == "fp64" else t.float()


def run(state):
    case, g = state["case"], state["g"]
    kind = case["kind"]
    if kind == "gradient":
        q, sigma, x = (state[k].detach().requires_grad_(True) for k in ("q", "sigma", "x"))
        F = M.free_energy(q, sigma, x, g)
        F.backward()
        return {"F": F.detach(), "q": q.grad, "sigma": sigma.grad, "x": x.grad}
    if kind == "hvp":
        return g.tangent(*state["tangent"])
    # new inputs of this pass
    g.q.copy_(state["q"])
    g.sigma.copy_(state["sigma"])
    g.x.copy_(state["x"])
    if kind == "run":
        g.build_neighbors()
        _, done = g.run_staggered(case["steps"], 1.0, 0.0, case["iters"], state["fire"])
        return {"done": done, "x": g.x, "q": _kept(case, g.q), "sigma": _kept(case, g.sigma)}
    if kind == "evaluate":
        g.build_neighbors()
        g.free_energy_grad()
        return {"F4": g.F4, "gq": _kept(case, g.gq), "gs": _kept(case, g.gs), "mu_ex": g.mu_ex, "mu": g.mu}
    g.build_neighbors()
    g.free_energy_grad(with_mu=False, asynchronous=True)
    g.diffuse_step(state["dt"], mu_ex=g.mu_ex, asynchronous=True)
    out = {"F4": g.F4, "gq": _kept(case, g.gq), "gs": _kept(case, g.gs), "mu_ex": g.mu_ex, "x": g.x}
    if kind == "step":
        out["iters"] = g.relax(0.0, case["iters"], state["fire"])[1]
        out["q"], out["sigma"] = _kept(case, g.q), _kept(case, g.sigma)
    else:
        g.sync_status()
    return out


# ------------------------------------------------------------------ work
def _sites(case):
    c = case.get("cells", 0)
    if case["system"] == "ensemble":
        m = (4 + case["cmax"]) / 2.0
        return int(4 * case["count"] * (m**3 + m * ((case["cmax"] - 3) ** 2 - 1) / 4.0))  # mean of the cubed uniform side
    return 8 * c * c * max(4, c // 2) if case["system"] == "slab" else 4 * c**3


def work(case):
    """Bytes: the state (q, sigma, x, T) in, the results out.  Operations:
    per evaluation and unordered pair inside the cut-off the 12 nodes of the
    rule with a distance, a switch and per radial term an exponential, a
    product and a sum (values; twice that with derivatives)."""
    n, S = _sites(case), 1 if case["system"] in ("vacancy", "vacancy_stable", "copper", "ensemble") else 2
    terms = {1: 2, 2: 5}[S] if case["system"] != "slab" else 4
    pairs = n * (60 if case["system"] == "slab" else 27)
    node = 12 + 4 * terms
    state = 8 * n * (5 + S)
    evals = {"evaluate": 1, "gradient": 1, "diffuse": 1, "hvp": 2}.get(case["kind"], 0)
    if case["kind"] in ("step", "run"):
        evals = case.get("steps", 1) * (case["iters"] + 2)
    out = 8 * n * {"evaluate": 4 + 2 * S, "gradient": 4 + S, "diffuse": 4 + 2 * S, "step": 8 + 2 * S, "run": 4 + S,
                   "hvp": 8 + 2 * S}[case["kind"]]
    flops = evals * pairs * 12 * 2 * node
    if case.get("embedding"):
        flops += pairs * 2 * 25 * 2 * 16
    return {"bytes": float(state + out), "flops": float(flops)}


# ------------------------------------------------------------------ the same in 64 bits
class _Radial:
    """The distinct radial terms of a potential and which species pair uses which."""

    def __init__(self, pot, params=None):
        self.S, self.rs, self.rc = pot.n_species, pot.r_switch, pot.r_cut
        terms, self.phi, self.f = [], {}, {}

        def add(A, kappa, lam):
            if A == 0.0:
                return None
            key = (math.log(A) + kappa, lam)
            if key not in terms:
                terms.append(key)
            return terms.index(key)

        for k in range(self.S):
            for l in range(k, self.S):
                if pot.cross_geomean and k != l:
                    u = add(math.sqrt(pot.phi_A[k, k] * pot.phi_A[l, l]), 0.5 * (pot.phi_p[k, k] + pot.phi_p[l, l]),
                            0.5 * (pot.phi_p[k, k] / pot.phi_r0[k, k] + pot.phi_p[l, l] / pot.phi_r0[l, l]))
                else:
                    u = add(pot.phi_A[k, l], pot.phi_p[k, l], pot.phi_p[k, l] / pot.phi_r0[k, l])
                self.phi[k, l] = self.phi[l, k] = u
        self.n_phi = len(terms)
        phi_terms, terms = terms, []
        for k in range(self.S):
            for l in range(self.S):
                v = add(pot.f_xi[k, l], pot.f_q[k, l], pot.f_q[k, l] / pot.f_r0[k, l])
                self.f[k, l] = None if v is None else self.n_phi + v
        self.terms = phi_terms + terms
        both = torch.tensor(self.terms, dtype=torch.float64, device=DEV).reshape(-1, 2)
        self.c, self.lam = both[:, 0].clone(), both[:, 1].clone()
        self.E = [float(e) for e in pot.E]

    def at(self, w, which):
        """{u: term u at squared distance w}."""
        r = torch.sqrt(w)
        t = ((r - self.rs) / (self.rc - self.rs)).clamp(0.0, 1.0)
        sw = 1.0 - t * t * t * (10.0 - t * (15.0 - 6.0 * t))
        return {u: torch.exp(self.c[u] - self.lam[u] * r) * sw for u in which}

    def used(self, table):
        return sorted({u for u in table.values() if u is not None})


def _lattice_pairs(nx, ny, nz, nb, basis, a, reach, open_z):
    """(i, j) of the unordered pairs of lattice sites within `reach`, a chunk at
    a time; site index ((sub, cell), b) as the recipes number them: host cells
    first, then octahedral cells."""
    cell = torch.arange(nx * ny * nz, device=DEV)
    ix, iy, iz = cell // (ny * nz), (cell // nz) % ny, cell % nz

    def site(c, b):
        return (b // 4) * (4 * nx * ny * nz) + 4 * c + b % 4

    buf, held = [], 0
    for b in range(nb):
        for b2 in range(nb):
            for dx in range(-2, 3):
                for dy in range(-2, 3):
                    for dz in range(-2, 3):
                        if (dx, dy, dz, b2) <= (0, 0, 0, b):
                            continue  # each unordered pair once
                        if np.linalg.norm((np.array([dx, dy, dz]) + basis[b2] - basis[b]) * a) > reach:
                            continue
                        j = ((ix + dx) % nx * ny + (iy + dy) % ny) * nz + (iz + dz) % nz
                        i = cell
                        if open_z:
                            ok = (iz + dz >= 0) & (iz + dz < nz)
                            i, j = i[ok], j[ok]
                        buf.append((site(i, b), site(j, b2)))
                        held += i.numel()
                        if held > 4_000_000:
                            yield tuple(torch.cat(t) for t in zip(*buf))
                            buf, held = [], 0
    if buf:
        yield tuple(torch.cat(t) for t in zip(*buf))


class _Exact:
    """The method in float64 torch on a concatenation of systems."""

    def __init__(self, case, systems):
        s0 = systems[0]
        self.case, self.S, self.s0 = case, s0.S, s0
        t = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device=DEV)  # noqa: E731
        self.q = t(np.concatenate([s.q for s in systems], axis=1))
        self.sigma = t(np.concatenate([s.sigma for s in systems]))
        self.x = t(np.concatenate([s.x for s in systems], axis=1))
        self.T = t(np.concatenate([s.T for s in systems]))
        self.n = self.sigma.numel()
        self.seg = torch.cat([torch.full((s.n,), b, device=DEV) for b, s in enumerate(systems)])
        self.nsys = len(systems)
        self.L = t(np.stack([s.L for s in systems], axis=1))
        self.R = _Radial(s0.pot)
        self.systems = systems
        self.kept = None

    def shape(self, s):
        if self.case["system"] == "slab":
            nx, ny = int(round(s.L[0] / s.a)), int(round(s.L[1] / s.a))
            return nx, ny, s.n // (8 * nx * ny), 8, np.concatenate([W.FCC_BASIS, W.OCTA_BASIS]), True
        nx = int(round(s.L[0] / s.a))
        return nx, nx, s.n // (4 * nx * nx), 4, W.FCC_BASIS, self.case["system"] == "surface"

    def chunks(self, reach=5.9):
        if self.kept is not None:
            yield from self.kept
            return
        kept, buf, held, at = [], [], 0, 0
        for s in self.systems:
            nx, ny, nz, nb, basis, open_z = self.shape(s)
            for i, j in _lattice_pairs(nx, ny, nz, nb, basis, s.a, reach, open_z):
                buf.append((i + at, j + at))
                held += i.numel()
                if held > 2_000_000:
                    c = tuple(torch.cat(v) for v in zip(*buf))
                    buf, held = [], 0
                    if self.n <= 1_200_000:
                        kept.append(c)
                    yield c
            at += s.n
        if buf:
            c = tuple(torch.cat(v) for v in zip(*buf))
            kept.append(c)
            yield c
        if self.n <= 1_200_000:
            self.kept = kept

    def separation(self, q, i, j):
        L = self.L[:, self.seg[i]]
        d = q[:, j] - q[:, i]
        return d - L * torch.round(d / L).detach()

    def averages(self, d, si, sj, which):
        """{u: sum over the 12 nodes / 12} of the terms `which` (App. A)."""
        D2 = (d * d).sum(0)
        acc = {u: 0.0 for u in which}
        for s in (SQRT6 * si, SQRT6 * sj):
            for a in range(3):
                for sign in (2.0, -2.0):
                    for u, v in self.R.at(D2 + s * s + sign * s * d[a], which).items():
                        acc[u] = acc[u] + v
        return {u: v / 12.0 for u, v in acc.items()}

    def embedding(self, rb, ra):
        """e, F', F'' of every species (Eq. F_taylor_mxe)."""
        e, F1, F2 = [], [], []
        for k in range(self.S):
            Ek = self.R.E[k]
            sq = torch.sqrt(rb[k])
            F1.append(-Ek / (2.0 * sq))
            F2.append(Ek / (4.0 * rb[k] * sq))
            e.append(-Ek * sq + F1[k] * (ra[k] - rb[k]))
        return e, F1, F2

    def mixing(self):
        x, T = self.x, self.T
        xv = 1.0 - x.sum(0)
        xlx = lambda v: torch.where(v > 0, v * torch.log(v.clamp_min(1e-300)), torch.zeros_like(v))  # noqa: E731
        return KB * T * (sum(xlx(x[k]) for k in range(self.S)) + xlx(xv)), xv

    def evaluate(self):
        """E_V, F_vib, F_mix, F per system; dF/dq, dF/dsigma, mu_ex, mu."""
        R, S, n = self.R, self.S, self.n
        fu, pu = R.used(R.f), R.used(R.phi)
        zero = lambda *sh: torch.zeros(sh, dtype=torch.float64, device=DEV)  # noqa: E731
        rb, ra = zero(S, n), zero(S, n)
        with torch.no_grad():
            for i, j in self.chunks():
                d = self.separation(self.q, i, j)
                st = R.at((d * d).sum(0), fu)
                av = self.averages(d, self.sigma[i], self.sigma[j], fu)
                for (k, l), v in R.f.items():
                    if v is None:
                        continue
                    rb[k].index_add_(0, i, self.x[l, j] * st[v])
                    rb[k].index_add_(0, j, self.x[l, i] * st[v])
                    ra[k].index_add_(0, i, self.x[l, j] * av[v])
                    ra[k].index_add_(0, j, self.x[l, i] * av[v])
        e, F1, F2 = self.embedding(rb, ra)
        a = [self.x[k] * F2[k] * (ra[k] - rb[k]) for k in range(S)]
        b = [self.x[k] * F1[k] for k in range(S)]
        gq, gs, mu, Es = zero(3, n), zero(n), zero(S, n), zero(n)
        for i, j in self.chunks():
            qi, qj = self.q[:, i].requires_grad_(True), self.q[:, j].requires_grad_(True)
            si, sj = self.sigma[i].requires_grad_(True), self.sigma[j].requires_grad_(True)
            L = self.L[:, self.seg[i]]
            d = qj - qi
            d = d - L * torch.round(d / L).detach()
            st = R.at((d * d).sum(0), fu)
            av = self.averages(d, si, sj, sorted(set(fu + pu)))
            V = 0.0
            for (k, l), u in R.phi.items():
                if u is not None:
                    w = self.x[k, i] * self.x[l, j]
                    V = V + w * av[u]
                    Es.index_add_(0, i, (0.5 * w * av[u]).detach())
                    Es.index_add_(0, j, (0.5 * w * av[u]).detach())
                    mu[k].index_add_(0, i, (self.x[l, j] * av[u]).detach())
                    mu[l].index_add_(0, j, (self.x[k, i] * av[u]).detach())
            for (k, l), v in R.f.items():
                if v is None:
                    continue
                V = V + (b[k][i] * self.x[l, j] + b[k][j] * self.x[l, i]) * av[v]
                V = V + (a[k][i] * self.x[l, j] + a[k][j] * self.x[l, i]) * st[v]
                mu[l].index_add_(0, i, (a[k][j] * st[v] + b[k][j] * av[v]).detach())
                mu[l].index_add_(0, j, (a[k][i] * st[v] + b[k][i] * av[v]).detach())
            g = torch.autograd.grad(V.sum(), (qi, qj, si, sj))
            gq.index_add_(1, i, g[0])
            gq.index_add_(1, j, g[1])
            gs.index_add_(0, i, g[2])
            gs.index_add_(0, j, g[3])
        for k in range(S):
            mu[k] += e[k]
            Es += self.x[k] * e[k]
        return self.finish(Es, gq, gs, mu)

    def finish(self, Es, gq, gs, mu):
        gs = gs - 3.0 * KB * self.T / self.sigma
        mix, xv = self.mixing()
        parts = torch.stack([Es, -3.0 * KB * self.T * torch.log(self.sigma), mix])
        F4 = torch.zeros((4, self.nsys), dtype=torch.float64, device=DEV)
        F4[:3].index_add_(1, self.seg, parts)
        F4[3] = F4[:3].sum(0)
        ln = lambda v: torch.log(v.clamp_min(1e-300))  # noqa: E731
        full = mu + KB * self.T * (ln(self.x) - ln(xv))
        return {"F4": F4[:, 0] if self.nsys == 1 else F4.T, "gq": gq, "gs": gs, "mu_ex": mu, "mu": full}

    def energy(self, q, sigma, x, exact_rule=False):
        """E_V as one differentiable scalar (small systems)."""
        R, S, n = self.R, self.S, self.n
        fu = R.used(R.f)
        E = 0.0
        rb, ra = [0.0] * S, [0.0] * S
        add = lambda i, v: torch.zeros(n, dtype=torch.float64, device=DEV).index_add(0, i, v)  # noqa: E731
        for i, j in self.chunks():
            d = self.separation(q, i, j)
            st = R.at((d * d).sum(0), fu)
            av = self.averages(d, sigma[i], sigma[j], range(len(R.terms)))
            for (k, l), u in R.phi.items():
                if u is not None:
                    E = E + (x[k, i] * x[l, j] * av[u]).sum()
            for (k, l), v in R.f.items():
                if v is not None and not exact_rule:
                    rb[k] = rb[k] + add(i, x[l, j] * st[v]) + add(j, x[l, i] * st[v])
                    ra[k] = ra[k] + add(i, x[l, j] * av[v]) + add(j, x[l, i] * av[v])
        if not exact_rule:
            e, _, _ = self.embedding(rb, ra)
            return E + sum((x[k] * e[k]).sum() for k in range(S))
        # App. A's rule over a site and its neighbours inside the cut-off:
        # N sites, every node moves one of them by sigma sqrt(3 N) along an axis
        ij = [c for c in self.chunks()]
        i = torch.cat([c[0] for c in ij] + [c[1] for c in ij])
        j = torch.cat([c[1] for c in ij] + [c[0] for c in ij])
        d = self.separation(q, i, j)
        D2 = (d * d).sum(0)
        inside = D2.detach() < R.rc**2
        i, j, d, D2 = i[inside], j[inside], d[:, inside], D2[inside]
        N = 1.0 + torch.bincount(i, minlength=n).to(torch.float64)
        hop = torch.sqrt(3.0 * N)
        st = R.at(D2, fu)
        for k in range(S):
            dens = lambda f: sum(x[l, j] * f[R.f[k, l]] for l in range(S) if R.f[k, l] is not None)  # noqa: E731
            at0 = dens(st)
            rho = add(i, at0)
            tot = 0.0
            for a in range(3):
                for sign in (2.0, -2.0):
                    own = hop[i] * sigma[i]
                    tot = tot + torch.sqrt(add(i, dens(R.at(D2 + own * own - sign * own * d[a], fu))))
                    its = hop[i] * sigma[j]
                    moved = dens(R.at(D2 + its * its + sign * its * d[a], fu))
                    tot = tot + add(i, torch.sqrt(rho[i] - at0 + moved))
            E = E + (x[k] * (-R.E[k]) * tot / (6.0 * N)).sum()
        return E

    def evaluate_rule(self):
        v = [t.clone().requires_grad_(True) for t in (self.q, self.sigma, self.x)]
        E = self.energy(*v, exact_rule=True)
        gq, gs, mu = torch.autograd.grad(E, v)
        Es = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        Es[0] = E.detach()
        return self.finish(Es, gq, gs, mu)

    def hvp(self, tangent):
        dq, ds, dx = (torch.as_tensor(t, device=DEV) for t in tangent)
        R = self.R
        R.c, R.lam = R.c.requires_grad_(True), R.lam.requires_grad_(True)
        v = [t.clone().requires_grad_(True) for t in (self.q, self.sigma, self.x)]
        E = self.energy(*v) - 3.0 * KB * (self.T * torch.log(v[1])).sum()
        every = v + [R.c, R.lam]
        g = torch.autograd.grad(E, every, create_graph=True)
        along = (g[0] * dq).sum() + (g[1] * ds).sum() + (g[2] * dx).sum()
        h = torch.autograd.grad(along, every)
        return {"gq": g[0].detach(), "gs": g[1].detach(), "mu_ex": g[2].detach(), "gq_t": h[0], "gs_t": h[1],
                "mu_ex_t": h[2], "dterm": torch.cat([g[3].detach(), g[4].detach(), h[3], h[4]])}

    # master equation and relaxation
    def bonds(self):
        s = self.s0
        r_bond = 0.5 * (s.a / math.sqrt(2.0) + s.a)
        sub = torch.cat([torch.as_tensor(t.sublattice, device=DEV) for t in self.systems])
        for i, j in self.chunks():
            d = self.separation(self.q, i, j)
            ok = ((d * d).sum(0) < r_bond**2) & (sub[i] == sub[j]) & (((s.mobile_mask >> sub[i].int()) & 1) == 1)
            if bool(ok.any()):
                yield i[ok], j[ok]

    def euler(self, mu, dt):
        """x after one forward-Euler step (Eq. MassTransport); dt per system."""
        x, T, s = self.x, self.T, self.s0
        D = s.nu0 * torch.exp(-s.Qm / (KB * T))
        xv = 1.0 - x.sum(0)
        rate = torch.zeros_like(x)
        for i, j in self.bonds():
            for k in range(self.S):
                dm = (mu[k, i] - mu[k, j]) / KB
                net = D[i] * x[k, i] * xv[j] * torch.exp(dm / T[i]) - D[j] * x[k, j] * xv[i] * torch.exp(-dm / T[j])
                rate[k].index_add_(0, i, -net)
                rate[k].index_add_(0, j, net)
        self.x = x + dt[self.seg] * rate

    def fire(self, iters):
        """`iters` FIRE updates of (q, sigma), each system with its own controls."""
        m = self.nsys
        full = lambda v: torch.full((m,), v, dtype=torch.float64, device=DEV)  # noqa: E731
        dt, alpha, n_pos = full(0.02), full(0.1), full(0.0)
        v = torch.zeros((4, self.n), dtype=torch.float64, device=DEV)
        total = lambda t: torch.zeros(m, dtype=torch.float64, device=DEV).index_add(0, self.seg, t.sum(0))  # noqa: E731
        for it in range(iters):
            g = self.evaluate()
            f = -torch.cat([g["gq"], g["gs"][None]])
            keep = full(1.0)
            if it > 0:
                up = total(f * v) > 0.0
                n_pos = torch.where(up, n_pos + 1.0, 0.0 * n_pos)
                grow = up & (n_pos > 5)
                dt = torch.where(up, torch.where(grow, (1.1 * dt).clamp_max(0.1), dt), 0.5 * dt)
                alpha = torch.where(up, torch.where(grow, 0.99 * alpha, alpha), full(0.1))
                keep = up.to(torch.float64)
            sg = self.seg
            v = keep[sg] * v + dt[sg] * f
            mix = alpha * torch.sqrt(total(v * v) / total(f * f))
            v = (1.0 - alpha)[sg] * v + mix[sg] * f
            self.q = self.q + dt[sg] * v[:3]
            self.sigma = self.sigma + dt[sg] * v[3]


def exact(case, seed):
    if _sites(case) > 1_200_000 or (case["kind"] == "run" and _sites(case) * case["steps"] > 500_000):
        return None
    systems = _host_systems(case, seed)
    X = _Exact(case, systems)
    kind = case["kind"]
    if kind == "hvp":
        return X.hvp(_tangent(systems[0], seed))
    if kind == "run":
        dts = torch.tensor([s.dt_default() for s in systems], dtype=torch.float64, device=DEV)
        for _ in range(case["steps"]):
            X.euler(X.evaluate()["mu_ex"], dts)
            X.fire(case["iters"])
        return {"done": None, "x": X.x, "q": X.q, "sigma": X.sigma}
    g = X.evaluate_rule() if case.get("embedding") else X.evaluate()
    if kind == "gradient":
        return {"F": g["F4"][3], "q": g["gq"], "sigma": g["gs"], "x": g["mu"]}
    if kind == "evaluate":
        return g
    X.euler(g["mu_ex"], torch.tensor([_dt(case, systems[0])], dtype=torch.float64, device=DEV))
    out = {"F4": g["F4"], "gq": g["gq"], "gs": g["gs"], "mu_ex": g["mu_ex"], "x": X.x}
    if kind == "step":
        X.fire(case["iters"])
        out |= {"iters": None, "q": X.q, "sigma": X.sigma}
    return out
