"""Performance cases of the framework: what its users run, from one operator
application on the smallest lattice to a benchmark-sized MD trajectory, each
through the public entry points of the package (Context and
PseudofermionAction). Lattices and couplings are those of the `workloads`
module and of the tests; a drawn case takes any size of the same ranges.

A case is a dict of plain values. `kind` selects the entry point:

  apply       Context.apply_M / apply_Mdag / apply_MMdag, complex64 or complex128
  cg          Context.solve_cg: plain FP64 CG (the correlators' solves)
  spcg        Context.solve_spcg: the FP32 CG alone
  fgmres      Context.solve_fgmres: mixed-precision solve
  action      PseudofermionAction forward and backward (autograd)
  batched     Context.solve_batched, mixed precision, uneven lattices
  trajectory  Context.md_trajectory: one HMC trajectory
  chains      Context.md_trajectory_batched: many chains in lockstep
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1804_07195_gb300 as hmc

DEV = "cuda"


def listed():
    return [
        # The smallest call: M on the 6x6, nt = 16 lattice, the field loaded once; launch latency.
        dict(name="m_f64_6x6x16", kind="apply", op="M", prec=64, n=6, m=6, nt=16, U=2.0, beta=4.0, ms=0.0,
             sigma=0.0, loaded=True),
        # M^dagger in FP64 on an odd lattice (the paper's 51 x 51 sheet) with a new field: one step of a
        # correlator or a force that is not part of a longer solve.
        dict(name="mdag_f64_51x51x64", kind="apply", op="Mdag", prec=64, n=51, m=51, nt=64, U=3.5, beta=8.0,
             ms=0.4, sigma=0.0, loaded=False),
        # The operator of the solves in FP64 on the largest lattice the paper simulates.
        dict(name="mmdag_f64_102x102x64", kind="apply", op="MMdag", prec=64, n=102, m=102, nt=64, U=3.8, beta=12.0,
             ms=0.1, sigma=0.0, loaded=True),
        # The same in FP32, shifted, on a lattice whose vectors do not fit the L2 cache.
        dict(name="mmdag_f32_306x306x64", kind="apply", op="MMdag", prec=32, n=306, m=306, nt=64, U=3.8, beta=12.0,
             ms=0.0, sigma=0.25, loaded=True),
        # Plain FP64 CG on the 36 x 36 lattice (the tight solves of correlators and of reference runs).
        dict(name="cg_f64_36x36x64", kind="cg", n=36, m=36, nt=64, U=3.5, beta=8.0, ms=0.0, sigma=0.0, tol=1e-10),
        # The FP32 CG alone on an odd lattice.
        dict(name="spcg_51x51x64", kind="spcg", n=51, m=51, nt=64, U=3.5, beta=8.0, ms=0.1, sigma=0.0, tol=1e-5),
        # One mixed-precision solve at full size with the paper's inner factor a = 5.
        dict(name="fgmres_102x102x64", kind="fgmres", n=102, m=102, nt=64, U=3.8, beta=12.0, ms=0.0, sigma=0.0,
             tol=1e-10, a=5.0),
        # Action and force through autograd on the 12 x 12 lattice with two Hasenbusch masses.
        dict(name="action_12x12x32", kind="action", n=12, m=12, nt=32, U=3.0, beta=6.0, masses="0.3,1.0", tol=1e-10),
        # Many independent systems of uneven lattices in one call, three shifts per lattice.
        dict(name="batched_16_lattices", kind="batched", count=16, lats="6,12,18,24,36", nts="16,32,48", U=3.0,
             beta=6.0, masses="0.1,0.5,2.0", tol=1e-10),
        # A trajectory on a small lattice, where a run makes very many of them.
        dict(name="trajectory_12x12x32", kind="trajectory", n=12, m=12, nt=32, U=3.0, beta=6.0, masses="0.3,1.0",
             nmd=6, ratios="2,1", tau=0.75, tol=1e-10, action_tol=1e-12, a=5.0),
        # Chains on small uneven lattices advanced in lockstep.
        dict(name="chains_8_lattices", kind="chains", count=8, lats="6,12,18,24", nts="16,32,48", U=3.0, beta=6.0,
             masses="0.1,0.5,2.0", nmd=4, ratios="2,1,1", tau=0.5, tol=1e-10, action_tol=1e-12),
        # The benchmark lattice: a fifth of a trajectory (all its parts, three Hasenbusch masses).
        dict(name="trajectory_102x102x64", kind="trajectory", n=102, m=102, nt=64, U=3.8, beta=12.0,
             masses="0.1,0.5,2.0", nmd=6, ratios="6,2,2", tau=0.2, tol=1e-10, action_tol=1e-12, a=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: every kind, sizes spread over the
    logarithm of their range, even and odd, n and m independent."""
    kind = rng.choice(["apply", "apply", "cg", "spcg", "fgmres", "action", "batched", "trajectory", "chains"])
    lat = lambda lo, hi: dict(n=_log_int(rng, lo, hi), m=_log_int(rng, lo, hi))
    phys = dict(U=round(rng.uniform(1.0, 4.0), 2), beta=round(rng.uniform(4.0, 8.0), 2))
    ms = rng.choice([0.0, round(rng.uniform(0.05, 2.0), 3)])
    if kind == "apply":
        return dict(kind=kind, op=rng.choice(["M", "Mdag", "MMdag"]), prec=rng.choice([32, 64]), **lat(3, 200),
                    nt=_log_int(rng, 8, 96), **phys, ms=ms, sigma=rng.choice([0.0, 0.25]),
                    loaded=rng.choice([True, False]))
    if kind == "cg":
        return dict(kind=kind, **lat(4, 48), nt=_log_int(rng, 16, 64), **phys, ms=ms, sigma=0.0,
                    tol=rng.choice([1e-8, 1e-10, 1e-12]))
    if kind == "spcg":
        return dict(kind=kind, **lat(6, 110), nt=_log_int(rng, 16, 64), **phys, ms=round(rng.uniform(0.1, 2.0), 3),
                    sigma=rng.choice([0.0, 0.04]), tol=1e-5)
    if kind == "fgmres":
        return dict(kind=kind, **lat(6, 100), nt=_log_int(rng, 16, 64), **phys, ms=ms, sigma=0.0, tol=1e-10,
                    a=rng.choice([1.0, 5.0]))
    if kind == "action":
        return dict(kind=kind, **lat(4, 40), nt=_log_int(rng, 16, 64), **phys,
                    masses=rng.choice(["", "0.5", "0.3,1.0"]), tol=1e-10)
    if kind == "batched":
        return dict(kind=kind, count=_log_int(rng, 4, 20), lats="5,6,9,12,18,24,33", nts="16,32,48", **phys,
                    masses=rng.choice(["0.1,0.5,2.0", "0.5"]), tol=1e-10)
    if kind == "chains":
        return dict(kind=kind, count=_log_int(rng, 2, 10), lats="5,6,9,12,18", nts="16,32", **phys,
                    masses=rng.choice(["0.3,1.0", "0.5"]), nmd=4, ratios="2,1", tau=0.5, tol=1e-10, action_tol=1e-12)
    return dict(kind=kind, **lat(5, 60), nt=_log_int(rng, 16, 64), **phys, masses="0.3,1.0", nmd=rng.choice([2, 4]),
                ratios="2,1", tau=0.5, tol=1e-10, action_tol=1e-12, a=rng.choice([1.0, 5.0]))


# --------------------------------------------------------------------------
# Inputs: phi ~ N(0, delta U), complex vectors with E|b|^2 = 1, pi ~ N(0, 1).


def _masses(case):
    return [float(v) for v in case.get("masses", "").split(",") if v]


class _Draw:
    """The inputs of one lattice in a fixed order, from one generator on the
    device (the same values in `prepare` and in `exact`)."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed) % (1 << 62))

    def real(self, n, sd=1.0):
        return torch.randn(n, dtype=torch.float64, device=DEV, generator=self.g) * sd

    def cplx(self, n):
        return torch.complex(self.real(n, math.sqrt(0.5)), self.real(n, math.sqrt(0.5)))


def _lattice(case):
    return hmc.Lattice(case["n"], case["m"], case["nt"], 1.0, case["U"], case["beta"])


def _uneven(case, seed):
    """The lattices of a batched case, drawn from its lists."""
    pick = np.random.Generator(np.random.PCG64(np.random.SeedSequence(case["count"])))
    ls = [int(v) for v in case["lats"].split(",")]
    nts = [int(v) for v in case["nts"].split(",")]
    out = []
    for _ in range(case["count"]):
        n = int(pick.choice(ls))
        nt = int(pick.choice(nts))
        out.append(hmc.Lattice(n, n, nt, 1.0, case["U"], case["beta"]))
    return out


def _inputs(case, seed):
    """Plain inputs of a case as a dict of device tensors."""
    d = _Draw(seed)
    kind = case["kind"]
    if kind in ("batched", "chains"):
        items = []
        for lat in _uneven(case, seed):
            N = lat.nsites
            it = dict(lat=lat, phi=d.real(N, math.sqrt(lat.delta * lat.U)))
            if kind == "batched":
                it["b"] = [d.cplx(N) for _ in _masses(case)]
            else:
                it["pi"] = d.real(N)
                it["rho"] = [d.cplx(N) for _ in range(len(_masses(case)) + 1)]
            items.append(it)
        return dict(items=items)
    lat = _lattice(case)
    N = lat.nsites
    out = dict(lat=lat, phi=d.real(N, math.sqrt(lat.delta * lat.U)))
    if kind in ("action", "trajectory"):
        out["pi"] = d.real(N)
        out["rho"] = [d.cplx(N) for _ in range(len(_masses(case)) + 1)]
    else:
        b = d.cplx(N)
        out["b"] = b.to(torch.complex64) if kind == "spcg" or case.get("prec") == 32 else b
    return out


def _md_opts(case, tol):
    return hmc.SolverOpts(tol=tol, a=case.get("a", 5.0))


def _integ(case):
    return hmc.Integrator(0, case["nmd"], tuple(int(v) for v in case["ratios"].split(",")), 0.193, case["tau"])


def prepare(case, seed):
    inp = _inputs(case, seed)
    kind = case["kind"]
    lat = inp["items"][0]["lat"] if "items" in inp else inp["lat"]
    st = dict(case=case, inp=inp, ctx=hmc.Context(lat))
    if kind == "apply":
        st["out"] = torch.empty_like(inp["b"])
        if case["loaded"]:
            st["ctx"].load_field(inp["phi"])
    elif kind == "action":
        # the pseudofermions of the action, as a program keeps them along a trajectory: the plain vectors rho
        st["phi"] = inp["phi"].clone().requires_grad_(True)
    return st


def run(st):
    case, inp, ctx = st["case"], st["inp"], st["ctx"]
    kind = case["kind"]
    if kind == "apply":
        phi = None if case["loaded"] else inp["phi"]
        if case["op"] == "M":
            return ctx.apply_M(phi, case["ms"], inp["b"], out=st["out"])
        if case["op"] == "Mdag":
            return ctx.apply_Mdag(phi, case["ms"], inp["b"], out=st["out"])
        return ctx.apply_MMdag(phi, case["ms"], inp["b"], sigma=case["sigma"], out=st["out"])
    if kind == "cg":
        return ctx.solve_cg(inp["phi"], case["ms"], inp["b"], sigma=case["sigma"], tol=case["tol"])[0]
    if kind == "spcg":
        return ctx.solve_spcg(inp["phi"], case["ms"], inp["b"], sigma=case["sigma"], tol=case["tol"])[0]
    if kind == "fgmres":
        return ctx.solve_fgmres(inp["phi"], case["ms"], inp["b"], sigma=case["sigma"], tol=case["tol"],
                                a=case["a"])[0]
    if kind == "action":
        S = hmc.PseudofermionAction.apply(st["phi"], ctx, _masses(case), inp["rho"], _md_opts(case, case["tol"]),
                                          True, -1)
        (g,) = torch.autograd.grad(S, st["phi"])
        return S.detach(), g
    if kind == "batched":
        systems = [dict(lattice=it["lat"], phi=it["phi"], ms=mu, sigma=0.0, b=b, x=torch.empty_like(b),
                        tol=case["tol"])
                   for it in inp["items"] for mu, b in zip(_masses(case), it["b"])]
        ctx.solve_batched(systems, mixed=True)
        return [s["x"] for s in systems]
    if kind == "trajectory":
        phi, pi = inp["phi"].clone(), inp["pi"].clone()
        H0, H1, _ = ctx.md_trajectory(phi, pi, _masses(case), inp["rho"], _integ(case), _md_opts(case, case["tol"]),
                                      _md_opts(case, case["action_tol"]))
        return phi, pi, H0, H1
    chains = [dict(lattice=it["lat"], phi=it["phi"].clone(), pi=it["pi"].clone(), rho=it["rho"])
              for it in inp["items"]]
    H0, H1, _ = ctx.md_trajectory_batched(chains, _masses(case), _integ(case), _md_opts(case, case["tol"]),
                                          _md_opts(case, case["action_tol"]))
    return [c["phi"] for c in chains], [c["pi"] for c in chains], list(H0), list(H1)


# --------------------------------------------------------------------------
# What a pass cannot do without.


def _sites(case):
    if case["kind"] in ("batched", "chains"):
        return sum(lat.nsites for lat in _uneven(case, 0))
    return _lattice(case).nsites


def _cg_iterations(nt, beta, ms, tol):
    """CG's own bound, sqrt(kappa)/2 ln(2/tol), with the spectrum of the free
    operator (lowest mode 4 sin^2(pi / 2 nt) at m_s = 0, raised by the mass;
    highest near 4)."""
    low = 4.0 * math.sin(math.pi / (2 * nt)) ** 2 + (beta / nt * ms) ** 2
    return 0.5 * math.sqrt((2.0 + beta / nt * 3.0) ** 2 / low) * math.log(2.0 / tol)


def work(case):
    """Bytes: every input read once, every output written once (a solve's
    iterations can stay on the chip). Flops: 22 per site and application of M
    or M^dagger, 64 per site and CG iteration, iterations by CG's bound."""
    kind = case["kind"]
    if kind == "apply":
        N = _sites(case)
        per = 20 if case["prec"] == 32 else 40
        return {"bytes": per * N, "flops": 22 * N * (2 if case["op"] == "MMdag" else 1)}
    if kind in ("cg", "spcg", "fgmres"):
        N = _sites(case)
        its = _cg_iterations(case["nt"], case["beta"], case["ms"], case["tol"])
        return {"bytes": (24 if kind == "spcg" else 40) * N, "flops": int(64 * N * its)}
    lats = _uneven(case, 0) if kind in ("batched", "chains") else [_lattice(case)]
    masses = _masses(case)
    nbytes = flops = 0
    for lat in lats:
        N = lat.nsites
        if kind == "batched":
            nbytes += (8 + 32 * len(masses)) * N
            flops += sum(64 * N * _cg_iterations(lat.nt, lat.beta, mu, case["tol"]) for mu in masses)
            continue
        lower = [0.0] + masses  # the operator of each term's solve
        if kind == "action":
            nbytes += (8 + 16 * len(lower) + 8) * N
            flops += sum(2 * 64 * N * _cg_iterations(lat.nt, lat.beta, mu, case["tol"]) for mu in lower)
            continue
        nbytes += (16 + 16 + 16 * len(lower)) * N
        steps = [case["nmd"] // int(r) for r in case["ratios"].split(",")][:len(masses)] + [case["nmd"]]
        for k, mu in enumerate(lower):
            # two forces per Omelyan step and the first, the start's solve (for chi) and the final action
            its = (2 * steps[k] + 1) * _cg_iterations(lat.nt, lat.beta, mu, case["tol"])
            its += 2 * _cg_iterations(lat.nt, lat.beta, mu, case["action_tol"])
            flops += 64 * N * its
    return {"bytes": int(nbytes), "flops": int(flops)}


def tolerance(case):
    """Measured against `exact` over several seeds and drawn cases, times
    about four. Applications: the rounding of the stencil. Solves: the residual
    tolerance amplified by the operator's small modes. Trajectories and
    forces: the errors of the solves inside."""
    kind = case["kind"]
    if kind == "apply":
        return {"rel": 5e-16, "max": 5e-15} if case["prec"] == 64 else {"rel": 5e-7, "max": 5e-6}
    if kind in ("cg", "fgmres"):
        return {"rel": 40.0 * case["tol"]}
    if kind in ("batched", "spcg"):
        return {"rel": 8.0 * case["tol"]}
    return {"rel": 4e-8}


# --------------------------------------------------------------------------
# The same results in 64 bits, plain torch: the operator by rolls of the
# (sublattice, t, j, i) array, its solves by CG with refinement.


class _Op:
    """M and M^dagger of the honeycomb lattice at one field (Eq. ferm_op of
    arXiv:1804.07195), anti-periodic in time."""

    def __init__(self, lat, phi):
        self.sh = (2, lat.nt, lat.m, lat.n)
        self.e = torch.exp(1j * phi.reshape(self.sh))
        self.dk, self.delta = lat.delta * lat.kappa, lat.delta
        self.first = torch.ones(lat.nt, 1, 1, dtype=torch.float64, device=phi.device)
        self.first[0] = -1.0  # hop t-1 -> t wraps at t = 0
        self.last = torch.ones_like(self.first)
        self.last[-1] = -1.0

    def _hop(self, a, b):
        """(sum over B neighbours of A cells, sum over A neighbours of B cells)"""
        return b + b.roll(1, 2) + b.roll(1, 1), a + a.roll(-1, 2) + a.roll(-1, 1)

    def M(self, ms, x):
        a, b = x.reshape(self.sh)
        ha, hb = self._hop(a, b)
        oa = -a + self.first * (self.e[0] - self.delta * ms) * a.roll(1, 0) - self.dk * ha
        ob = b - self.last * (self.e[1].conj() - self.delta * ms) * b.roll(-1, 0) - self.dk * hb
        return torch.stack([oa, ob]).reshape(-1)

    def Mdag(self, ms, x):
        a, b = x.reshape(self.sh)
        ha, hb = self._hop(a, b)
        oa = -a + ((self.first * (self.e[0].conj() - self.delta * ms)) * a).roll(-1, 0) - self.dk * ha
        ob = b - ((self.last * (self.e[1] - self.delta * ms)) * b).roll(1, 0) - self.dk * hb
        return torch.stack([oa, ob]).reshape(-1)

    def A(self, ms, sigma, x):
        y = self.M(ms, self.Mdag(ms, x))
        return y + sigma * x if sigma else y

    def solve(self, ms, sigma, b):
        """(M M^dagger + sigma)^{-1} b: CG to 1e-8, refined once."""
        x = self._cg(ms, sigma, b, 1e-8)
        return x + self._cg(ms, sigma, b - self.A(ms, sigma, x), 1e-8)

    def _cg(self, ms, sigma, b, tol):
        x, r, p = torch.zeros_like(b), b.clone(), b.clone()
        rr = torch.vdot(r, r).real
        stop = tol * tol * float(rr)
        for it in range(20000):
            if it % 20 == 0 and float(rr) <= stop:
                break
            q = self.A(ms, sigma, p)
            alpha = rr / torch.vdot(p, q).real
            x += alpha * p
            r -= alpha * q
            new = torch.vdot(r, r).real
            p = r + (new / rr) * p
            rr = new
        return x

    def dforce(self, eta, w):
        """-2 Re(conj(eta) dM w): dM/dphi in row (x, t) is i s e^{+-i phi} towards the time partner."""
        ea, eb = eta.reshape(self.sh)
        wa, wb = w.reshape(self.sh)
        fa = -2.0 * (ea.conj() * 1j * self.first * self.e[0] * wa.roll(1, 0)).real
        fb = -2.0 * (eb.conj() * 1j * self.last * self.e[1].conj() * wb.roll(-1, 0)).real
        return torch.stack([fa, fb]).reshape(-1)


class _Terms:
    """The Hasenbusch terms (Section 5.1) at fixed chi."""

    def __init__(self, lat, masses, chis):
        self.lat, self.masses, self.chis = lat, masses, chis
        self.lower = [0.0] + list(masses)
        self.inv = 1.0 / (lat.delta * lat.U)

    def _eta(self, op, i):
        src = self.chis[i] if i == len(self.masses) else op.M(self.masses[i], self.chis[i])
        eta = op.solve(self.lower[i], 0.0, src)
        return src, eta

    def grad(self, phi, i):
        op = _Op(self.lat, phi)
        _, eta = self._eta(op, i)
        w = op.Mdag(self.lower[i], eta)
        if i < len(self.masses):
            w = w - self.chis[i]
        return op.dforce(eta, w)

    def action(self, phi):
        op = _Op(self.lat, phi)
        S = 0.5 * self.inv * float(torch.dot(phi, phi))
        for i in range(len(self.chis)):
            src, eta = self._eta(op, i)
            S += float(torch.vdot(src, eta).real)
        return S


def _trajectory(lat, phi, pi, masses, rho, case):
    """Nested Omelyan (Section 5.2), force first, each force evaluated once per field."""
    op = _Op(lat, phi)
    lower = [0.0] + list(masses)
    chis = [op.Mdag(mu, op.solve(mu, 0.0, op.M(lower[i], rho[i]))) for i, mu in enumerate(masses)]
    chis.append(op.M(lower[-1], rho[-1]))
    T = _Terms(lat, masses, chis)
    H0 = 0.5 * T.inv * float(torch.dot(phi, phi)) + 0.5 * float(torch.dot(pi, pi))
    H0 += sum(float(torch.vdot(r, r).real) for r in rho)
    n = len(masses)
    ratios = [int(v) for v in case["ratios"].split(",")][:n]
    steps = [case["nmd"] // r for r in ratios] + [case["nmd"]]
    mult = [steps[0]] + [steps[k] // steps[k - 1] for k in range(1, n + 1)]
    zeta = 0.193
    s = dict(phi=phi.clone(), pi=pi.clone(), ver=0, cache={})

    def P(k, c):
        if s["cache"].get(k, (None, -1))[1] != s["ver"]:
            g = T.grad(s["phi"], k)
            s["cache"][k] = (g + T.inv * s["phi"] if k == n else g, s["ver"])
        s["pi"] = s["pi"] - c * s["cache"][k][0]

    def inner(k, h, second):
        if k == n:
            s["phi"] = s["phi"] + 0.5 * h * s["pi"]
            s["ver"] += 1
            return
        r, hh = mult[k + 1], h / mult[k + 1]
        if second and r % 2:
            P(k + 1, 0.5 * (1.0 - 2.0 * zeta) * hh)
            inner(k + 1, hh, True)
            P(k + 1, zeta * hh)
        for _ in range(r // 2):
            step(k + 1, hh)
        if not second and r % 2:
            P(k + 1, zeta * hh)
            inner(k + 1, hh, False)
            P(k + 1, 0.5 * (1.0 - 2.0 * zeta) * hh)

    def step(k, h):
        P(k, zeta * h)
        inner(k, h, False)
        P(k, (1.0 - 2.0 * zeta) * h)
        inner(k, h, True)
        P(k, zeta * h)

    for _ in range(steps[0]):
        step(0, case["tau"] / steps[0])
    H1 = T.action(s["phi"]) + 0.5 * float(torch.dot(s["pi"], s["pi"]))
    return s["phi"], s["pi"], H0, H1


def _exact_seconds(case):
    """Rough time of `exact`: about 1.1 ms per iteration of the bound on lattices of these sizes."""
    kind = case["kind"]
    if kind == "apply":
        return 0.1
    lats = _uneven(case, 0) if kind in ("batched", "chains") else [_lattice(case)]
    masses = _masses(case)
    t = 0.0
    for lat in lats:
        its = lambda mu: 2 * _cg_iterations(lat.nt, lat.beta, mu, 1e-8)
        if kind in ("cg", "spcg", "fgmres"):
            t += its(case["ms"])
        elif kind == "batched":
            t += sum(its(mu) for mu in masses)
        elif kind == "action":
            t += 2 * sum(its(mu) for mu in [0.0] + masses)
        else:
            steps = [case["nmd"] // int(r) for r in case["ratios"].split(",")][:len(masses)] + [case["nmd"]]
            t += sum((2 * st + 3) * its(mu) for st, mu in zip(steps, [0.0] + masses))
    return 1.1e-3 * t


def exact(case, seed):
    if _exact_seconds(case) > 22.0:
        return None
    inp = _inputs(case, seed)
    kind = case["kind"]
    if kind == "apply":
        op, x = _Op(inp["lat"], inp["phi"]), inp["b"].to(torch.complex128)
        if case["op"] == "MMdag":
            return op.A(case["ms"], case["sigma"], x)
        return (op.M if case["op"] == "M" else op.Mdag)(case["ms"], x)
    if kind in ("cg", "spcg", "fgmres"):
        return _Op(inp["lat"], inp["phi"]).solve(case["ms"], case["sigma"], inp["b"].to(torch.complex128))
    if kind == "action":
        T = _Terms(inp["lat"], _masses(case), inp["rho"])
        S = torch.tensor(T.action(inp["phi"]), dtype=torch.float64, device=DEV)
        return S, sum(T.grad(inp["phi"], i) for i in range(len(inp["rho"]))) + T.inv * inp["phi"]
    if kind == "batched":
        return [_Op(it["lat"], it["phi"]).solve(mu, 0.0, b)
                for it in inp["items"] for mu, b in zip(_masses(case), it["b"])]
    if kind == "trajectory":
        return _trajectory(inp["lat"], inp["phi"], inp["pi"], _masses(case), inp["rho"], case)
    outs = [_trajectory(it["lat"], it["phi"], it["pi"], _masses(case), it["rho"], case) for it in inp["items"]]
    return [o[0] for o in outs], [o[1] for o in outs], [o[2] for o in outs], [o[3] for o in outs]
