"""The work that users of this library have it do, as cases that can be timed and checked.

A case is one call sequence of a flow solver or a calibration loop on a field of points: the
rates and transport of a time step, the exact Jacobian products of an implicit stage, the
gradients of a calibration, a whole implicit reactor step, or fields that live in host memory.
Mechanisms are the synthetic ones of this package's ``synth`` module (9, 53 and 120 species, or
others drawn by the same generator); points are grouped like a spectral-element mesh of order 7
(512 points per element), with ragged counts beside whole elements.
"""
import math

import numpy as np
import torch

import paper_2409_06404_gb300 as nk
from paper_2409_06404_gb300 import synth

RU = 8.314462618
P0 = 101325.0
EL = 512                       # points of an element of order 7
DIRECTIONS = 10                # Krylov directions per implicit-stage linearization

H2 = dict(K=9, R=21, n_tb=3, n_troe=1, mech_seed=1009)
CH4 = dict(K=53, R=325, n_tb=20, n_troe=25, mech_seed=1053)
BIG = dict(K=120, R=700, n_tb=40, n_troe=60, mech_seed=1120)


def listed():
    return [
        # one element on its own: what a solver calls for a probe, a small rank or a test, where
        # launches and latency are everything
        dict(name="element_h2", path="forward", n=EL, precision="fp64", **H2),
        # a small box with the hydrogen mechanism (64 elements): rates and properties of a step
        dict(name="box_h2", path="forward", n=64 * EL, precision="fp64", **H2),
        # production field, methane-sized mechanism: the rates kernel of a step
        dict(name="rates_ch4", path="rates", n=4096 * EL, precision="fp64", **CH4),
        # the same field's transport properties
        dict(name="transport_ch4", path="transport", n=4096 * EL, precision="fp64", **CH4),
        # large mechanism in the mixed form: rates and properties of a step
        dict(name="forward_big_mixed", path="forward", n=216 * EL, precision="mixed", **BIG),
        # an exact Jacobian-vector product of the rates, recomputed (no stored data)
        dict(name="jvp_ch4", path="jvp", n=1000 * EL, precision="fp64", **CH4),
        # calibration: loss gradient of (T, Y, ln A) through autograd, ragged batch of states
        dict(name="train_ch4", path="train", n=200003, precision="fp64", **CH4),
        # Newton-Krylov stage: one linearization with the rates, ten exact products from it
        dict(name="stage_ch4", path="stage", n=512 * EL, precision="fp64", **CH4),
        # the same with the single-precision data that a float Krylov basis takes
        dict(name="stage_f32_ch4", path="stage_f32", n=343 * EL, precision="f32", **CH4),
        # implicit Euler step with the block-Jacobi preconditioner on burnt-gas states
        dict(name="reactor_ch4", path="reactor", n=32 * EL, precision="fp64", **CH4),
        # thermodynamics and diffusion fluxes of a step
        dict(name="fluxes_ch4", path="fluxes", n=1728 * EL, precision="fp64", **CH4),
        # a CPU code that offloads rates and properties: page-locked host fields in and out
        dict(name="host_ch4", path="host", n=300000, precision="fp64", **CH4),
    ]


# ------------------------------------------------------------------------------- drawn cases
def _units(path, K, R):
    """Rough cost per point of a path, for the bound on a drawn case's size."""
    rates, trans = 60.0 * R, 8.0 * K * K + 40.0 * K
    return {"rates": rates, "transport": trans, "forward": rates + trans, "jvp": 2 * rates, "train": 3.5 * rates,
            "stage": 2.5 * rates + DIRECTIONS * rates, "stage_f32": 4 * rates + DIRECTIONS * 0.6 * rates,
            "reactor": 2.0 * (K + 1) ** 3, "fluxes": 200.0 * K, "host": 2 * (rates + trans)}[path]


def draw(rng):
    path = rng.choice(["forward", "forward", "rates", "transport", "jvp", "train", "stage", "stage_f32", "reactor",
                       "fluxes", "host"])
    if path == "reactor" or rng.random() < 0.5:
        m = dict(CH4) if path == "reactor" else dict(rng.choice([H2, CH4, CH4, BIG]))
    else:                                                   # another mechanism of the same family
        K = int(round(math.exp(rng.uniform(math.log(9), math.log(120)))))
        R = int(K * rng.uniform(2.5, 6.5))
        m = dict(K=K, R=R, n_tb=max(1, R // 16), n_troe=max(1, R // 13), mech_seed=rng.randrange(1, 10 ** 6))
    most = 4096 * EL * _units("rates", CH4["K"], CH4["R"]) / _units(path, m["K"], m["R"])
    most = min(most, 4096 * EL)
    if path in ("stage", "stage_f32"):
        most = min(most, 512 * EL)
    if path == "reactor":
        most = 32 * EL
    n = int(round(math.exp(rng.uniform(math.log(EL), math.log(max(most, 2 * EL))))))
    if rng.random() < 0.5:
        n = max(EL, n // EL * EL)                           # whole elements, else a ragged count
    precision = "f32" if path == "stage_f32" else "fp64"
    if path in ("forward", "rates", "transport", "host") and rng.random() < 0.35:
        precision = "mixed"
    return dict(path=path, n=n, precision=precision, **m)


# ------------------------------------------------------------------------------- inputs
_MECHS = {}


def _mechanism(case):
    """The mechanism's arrays on the host (what a user's program read from its mechanism file)."""
    key = tuple(case[k] for k in ("K", "R", "n_tb", "n_troe", "mech_seed"))
    if key not in _MECHS:
        K, R, n_tb, n_troe, seed = key
        elements = ("H", "O", "N") if K < 20 else ("C", "H", "O", "N")
        _MECHS[key] = synth.make_mechanism(K, R, n_tb, n_troe, elements=elements, seed=seed)
    return _MECHS[key]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _flame(case, seed):
    """T over a flame profile (300 to 2200 K with 5% noise), 1 atm, Dirichlet(0.3) mass fractions."""
    K, n, g = case["K"], case["n"], _gen(seed)
    f = dict(dtype=torch.float64, device="cuda")
    x = (torch.arange(n, **f) + 0.5) / n
    T = 300.0 + 950.0 * (1.0 + torch.tanh((x - 0.5) / 0.05))
    T = (T * (1.0 + 0.05 * torch.randn(n, generator=g, **f))).clamp_(300.0, 3500.0)
    Y = torch._standard_gamma(torch.full((K, n), 0.3, **f), generator=g)
    Y /= Y.sum(0)
    return T, torch.full((n,), P0, **f), Y


def _direction(case, seed, j):
    g = _gen(seed * 1000 + 17 + j)
    f = dict(dtype=torch.float64, device="cuda", generator=g)
    return torch.randn(case["n"], **f), torch.randn((case["K"], case["n"]), **f)


def _burnt(case, seed):
    """Chemical equilibria at 512 temperatures in 1300..2600 K (from element potentials), tiled
    over the points and perturbed by 1e-3 in Y and about 1 K in T: gas behind a flame."""
    mech, K, n, nu = _mechanism(case), case["K"], case["n"], 512
    rng = np.random.default_rng(case["mech_seed"] + 5000)
    Tu = np.linspace(1300.0, 2600.0, nu)
    a = np.where((Tu[None, :] <= mech.T_mid[:, None])[:, None, :], mech.nasa_lo[:, :, None], mech.nasa_hi[:, :, None])
    h = sum(a[:, j] * Tu ** j / (j + 1) for j in range(5)) + a[:, 5] / Tu
    s = a[:, 0] * np.log(Tu) + sum(a[:, j] * Tu ** j / j for j in range(1, 5)) + a[:, 6]
    gRT = h - s
    at = mech.atoms.astype(float)
    lam = np.linalg.lstsq(np.hstack([at, np.ones((K, 1))]), gRT, rcond=None)[0][:-1]
    base = -gRT + at @ (lam + 0.5 * rng.standard_normal(lam.shape))
    na = at.sum(axis=1)[:, None]
    lo, hi = np.full(nu, -1e4), np.full(nu, 1e4)
    for _ in range(200):
        t = 0.5 * (lo + hi)
        z = base + t[None, :] * na
        zm = z.max(axis=0)
        big = zm + np.log(np.exp(z - zm).sum(axis=0)) > 0.0
        hi, lo = np.where(big, t, hi), np.where(big, lo, t)
    Y = np.exp(base + 0.5 * (lo + hi)[None, :] * na) * mech.W[:, None]
    Y /= Y.sum(axis=0)
    g = _gen(seed)
    f = dict(dtype=torch.float64, device="cuda")
    idx = torch.arange(n, device="cuda") % nu
    T = torch.tensor(Tu, **f)[idx] + torch.randn(n, generator=g, **f)
    Yt = torch.tensor(Y, **f)[:, idx] * (1.0 + 1e-3 * torch.randn((K, n), generator=g, **f))
    Yt /= Yt.sum(0)
    return T, torch.full((n,), P0, **f), Yt.contiguous()


def _grad_x(case, seed):
    return 100.0 * torch.randn((3, case["K"], case["n"]), generator=_gen(seed * 1000 + 7), dtype=torch.float64,
                               device="cuda")


def _dmix(case, seed):
    u = torch.rand((case["K"], case["n"]), generator=_gen(seed * 1000 + 8), dtype=torch.float64, device="cuda")
    return 1e-5 * (1.0 + 99.0 * u)


def _dlnA(case, seed):
    return 0.1 * torch.randn(case["R"], generator=_gen(seed * 1000 + 9), dtype=torch.float64, device="cuda")


def prepare(case, seed):
    path = case["path"]
    T, p, Y = _burnt(case, seed) if path == "reactor" else _flame(case, seed)
    s = dict(case=case, m=nk.mechanism_load(_mechanism(case)), T=T, p=p, Y=Y)
    if path == "jvp":
        s["v"] = _direction(case, seed, 0)
    if path in ("stage", "stage_f32"):
        s["v"] = [_direction(case, seed, j) for j in range(DIRECTIONS)]
        # the stage's linearization storage, kept from step to step
        if path == "stage":
            s["lin"] = torch.empty((nk.linearization_slots_compact(s["m"]), case["n"]), dtype=torch.float64, device="cuda")
        else:
            s["lin"] = torch.empty((nk.linearization_slots_f32(s["m"]), case["n"]), dtype=torch.float32, device="cuda")
    if path == "train":
        s["dlnA"] = _dlnA(case, seed)
        s["bar"] = _direction(case, seed, 0)
    if path == "fluxes":
        s["D"], s["gradX"] = _dmix(case, seed), _grad_x(case, seed)
    if path == "reactor":
        s["opts"] = nk.reactor_opts(rtol=1e-6, atol_T=1e-6, atol_Y=1e-12, newton_tol=1e-4, lin_tol=1e-6,
                                    max_newton=20, krylov_dim=10, precond=1)
        s["ws"] = torch.empty(nk.reactor_workspace(s["m"], case["n"], 10, 1, 0), dtype=torch.uint8, device="cuda")
    if path == "host":
        s["host"] = [t.cpu().pin_memory() for t in (T, p, Y)]
        s["ws"] = torch.empty(nk.host_eval_workspace(s["m"], min(65536, case["n"])), dtype=torch.uint8, device="cuda")
        n, K = case["n"], case["K"]
        s["out"] = tuple(torch.empty(sh, dtype=torch.float64, pin_memory=True) for sh in ((K, n), (n,), (n,), (n,), (K, n)))
        del s["T"], s["p"], s["Y"]
    return s


# ------------------------------------------------------------------------------- one pass
def run(s):
    case, m = s["case"], s["m"]
    path, prec = case["path"], case["precision"]
    if path == "host":
        return nk.host_eval(m, *s["host"], precision=prec, chunk=65536, workspace=s["ws"], outputs=s["out"])
    T, p, Y = s["T"], s["p"], s["Y"]
    if path == "rates":
        return nk.rates_eval(m, T, p, Y, precision=prec)
    if path == "transport":
        return nk.transport_eval(m, T, p, Y, precision=prec)
    if path == "forward":
        return nk.rates_eval(m, T, p, Y, precision=prec), nk.transport_eval(m, T, p, Y, precision=prec)
    if path == "jvp":
        return nk.rates_jvp(m, T, p, Y, *s["v"])
    if path == "train":
        Tg, Yg, Ag = T.detach().requires_grad_(), Y.detach().requires_grad_(), s["dlnA"].detach().requires_grad_()
        omega, hrr = nk.rates(m, Tg, p, Yg, Ag)
        grads = torch.autograd.grad((omega, hrr), (Tg, Yg, Ag), grad_outputs=(s["bar"][1], s["bar"][0]))
        return omega.detach(), hrr.detach(), grads
    if path == "stage":
        lin, omega, hrr = nk.rates_linearize_compact(m, T, p, Y, lin=s["lin"], primal=True)
        return omega, hrr, [nk.rates_jvp_linearized_compact(m, T, p, Y, lin, *v) for v in s["v"]]
    if path == "stage_f32":
        fT, fY = nk.rhs_eval(m, T, p, Y)
        lin = nk.rates_linearize_f32(m, T, p, Y, lin=s["lin"])
        return fT, fY, [nk.rhs_jvp_linearized_f32(m, T, p, Y, lin, fT, fY, *v) for v in s["v"]]
    if path == "reactor":
        T1, Y1 = T.clone(), Y.clone()           # the step works in place: the caller keeps the old state
        nk.reactor_step(m, T1, p, Y1, 1e-5, s["opts"], workspace=s["ws"])
        return T1, Y1
    if path == "fluxes":
        return nk.thermo_eval(m, T, p, Y), nk.diffusion_fluxes(m, T, p, Y, s["D"], s["gradX"])
    raise KeyError(path)


# ------------------------------------------------------------------------------- what it cannot do without
def work(case):
    """Each input read once and each output written once; operations of the definitions (counted
    on the 53-species mechanism: about 67 per reaction for the rates, 24 per species pair for
    transport, each transcendental function as ten)."""
    K, R, n, path = case["K"], case["R"], case["n"], case["path"]
    state, out = 8 * (K + 2), 8 * (K + 1)
    fr, ft = 120.0 * R, 50.0 * K * K
    tr = 8 * (K + 2)
    nb, fl = {
        "rates": (state + out, fr),
        "transport": (state + tr, ft),
        "forward": (state + out + tr, fr + ft),
        "host": (state + out + tr, fr + ft),
        "jvp": (state + 2 * out, 2.0 * fr),
        "train": (state + 3 * out, 4.0 * fr),
        "stage": (state + out + DIRECTIONS * 2 * out, 2.0 * fr + DIRECTIONS * 30.0 * R),
        "stage_f32": (state + out + DIRECTIONS * 2 * out, 3.0 * fr + DIRECTIONS * 30.0 * R),
        "reactor": (state + out, 3.0 * fr + 2.0 / 3.0 * (K + 1) ** 3),
        "fluxes": (state + 8 * (4 + 3 * K) + 8 * (K + 6 * K + 6), 60.0 * K),
    }[path]
    return {"bytes": float(n) * nb, "flops": float(n) * fl}


# ------------------------------------------------------------------------------- the same in plain torch, 64 bits
class _Plain:
    """The definitions over torch tensors: T [n], p [n], Y [K, n] to outputs per point."""

    def __init__(self, mech):
        f = dict(dtype=torch.float64, device="cuda")
        t = lambda a: torch.tensor(np.asarray(a), **f)                                            # noqa: E731
        K, R = mech.K, mech.R
        self.K, self.R, self.p_ref = K, R, mech.p_ref
        self.W, self.lo, self.hi, self.Tm = t(mech.W), t(mech.nasa_lo), t(mech.nasa_hi), t(mech.T_mid)
        self.lnA, self.beta, self.Ea = t(mech.lnA), t(mech.beta), t(mech.Ea)
        self.tb = torch.tensor(np.flatnonzero(mech.rtype == 1), device="cuda")
        self.fo = torch.tensor(np.flatnonzero(mech.rtype == 2), device="cuda")
        fo = np.flatnonzero(mech.rtype == 2)
        self.lnA0, self.beta0, self.Ea0, self.troe = t(mech.lnA0[fo]), t(mech.beta0[fo]), t(mech.Ea0[fo]), t(mech.troe[fo])
        self.eff_tb, self.eff_fo = t(mech.eff[mech.rtype == 1]), t(mech.eff[fo])
        nr, npr = np.zeros((R, K)), np.zeros((R, K))
        sides = []
        for ptr, sp, nu, N in ((mech.reac_ptr, mech.reac_sp, mech.reac_nu, nr), (mech.prod_ptr, mech.prod_sp, mech.prod_nu, npr)):
            idx = np.full((R, 12), K)                                  # K: a row of ones
            for r in range(R):
                flat = [k for e in range(ptr[r], ptr[r + 1]) for k in [sp[e]] * nu[e]]
                idx[r, :len(flat)] = flat
                for k in flat:
                    N[r, k] += 1.0
            width = int(max(1, (idx < K).sum(axis=1).max()))
            sides.append(torch.tensor(idx[:, :width].copy(), device="cuda"))
        self.reac, self.prod = sides
        self.net = t(npr - nr)
        self.mu_fit, self.lam_fit = t(mech.mu_fit), t(mech.lam_fit)
        D = np.zeros((K, K, 4))
        i, j = np.triu_indices(K, 1)
        D[i, j] = mech.D_fit
        D[j, i] = mech.D_fit
        self.D_fit = t(D)

    def thermo(self, T):
        a = torch.where((T[None, :] <= self.Tm[:, None])[:, None, :], self.lo[:, :, None], self.hi[:, :, None])
        cp = sum(a[:, j] * T ** j for j in range(5))
        h = sum(a[:, j] * T ** j / (j + 1) for j in range(5)) + a[:, 5] / T
        s = a[:, 0] * torch.log(T) + sum(a[:, j] * T ** j / j for j in range(1, 5)) + a[:, 6]
        return cp, h, h - s

    def mixture(self, T, p, Y):
        Wbar = 1.0 / (Y / self.W[:, None]).sum(0)
        rho = p * Wbar / (RU * T)
        return Wbar, rho, rho * Y / self.W[:, None], Y * Wbar / self.W[:, None]

    def rates(self, T, p, Y, dlnA=None):
        _, rho, C, _ = self.mixture(T, p, Y)
        cp, h, g = self.thermo(T)
        lnT, shift = torch.log(T), 0.0 if dlnA is None else dlnA[:, None]
        lnk = self.lnA[:, None] + shift + self.beta[:, None] * lnT - (self.Ea / RU)[:, None] / T
        lnKc = -(self.net @ g) + self.net.sum(1)[:, None] * torch.log(P0 / (RU * T))
        k = torch.exp(lnk)
        if len(self.fo):
            sh0 = 0.0 if dlnA is None else dlnA[self.fo][:, None]
            k0 = torch.exp(self.lnA0[:, None] + sh0 + self.beta0[:, None] * lnT - (self.Ea0 / RU)[:, None] / T)
            Pr = k0 * (self.eff_fo @ C) / k[self.fo]
            a, T3, T1, T2 = (self.troe[:, j:j + 1] for j in range(4))
            Fc = (1 - a) * torch.exp(-T / T3) + a * torch.exp(-T / T1) + torch.where(T2 > 0, torch.exp(-T2 / T), torch.zeros_like(T))
            lF = torch.log10(Fc)
            u = torch.log10(Pr) - 0.4 - 0.67 * lF
            f1 = u / (0.75 - 1.27 * lF - 0.14 * u)
            k = k.index_copy(0, self.fo, k[self.fo] * Pr / (1 + Pr) * 10.0 ** (lF / (1 + f1 * f1)))
        C1 = torch.cat([C, torch.ones_like(C[:1])])
        side = lambda idx: torch.stack([C1[idx[:, e]] for e in range(idx.shape[1])]).prod(0)      # noqa: E731
        q = k * side(self.reac) - k * torch.exp(-lnKc) * side(self.prod)
        if len(self.tb):
            q = q.index_copy(0, self.tb, q[self.tb] * (self.eff_tb @ C))
        omega = self.net.T @ q
        return omega, -(RU * T) * (h * omega).sum(0)

    def sources(self, T, p, Y):
        omega, hrr = self.rates(T, p, Y)
        _, rho, _, _ = self.mixture(T, p, Y)
        cp = (Y * RU * self.thermo(T)[0] / self.W[:, None]).sum(0)
        return hrr / (rho * cp), self.W[:, None] * omega / rho

    def transport(self, T, p, Y):
        Wbar, _, _, X = self.mixture(T, p, Y)
        L = torch.log(T)
        poly = lambda c: c[..., 0:1] + L * (c[..., 1:2] + L * (c[..., 2:3] + L * c[..., 3:4]))    # noqa: E731
        mu_k, lam_k = torch.exp(poly(self.mu_fit)), torch.exp(poly(self.lam_fit))
        W = self.W
        mu = torch.zeros_like(T)
        D = torch.empty_like(Y)
        for k in range(self.K):
            t = 1 + torch.sqrt(mu_k[k] / mu_k) * ((W / W[k]) ** 0.25)[:, None]
            phi = (1 / (8 * (1 + W[k] / W)).sqrt())[:, None] * t * t
            mu = mu + X[k] * mu_k[k] / (X * phi).sum(0)
            den = X * torch.exp(-poly(self.D_fit[k])) * (p / self.p_ref)
            den[k] = 0.0
            XW = X * W[:, None]
            XW[k] = 0.0
            D[k] = XW.sum(0) / (Wbar * den.sum(0))
        return mu, 0.5 * ((X * lam_k).sum(0) + 1 / (X / lam_k).sum(0)), D

    def fluxes(self, T, p, Y, D, gradX):
        Wbar, rho, _, X = self.mixture(T, p, Y)
        cp, h, g = self.thermo(T)
        molar = {"cp_k": RU * cp, "h_k": RU * T * h, "g_k": RU * T * g}
        mass = {"cp_mix": (Y * molar["cp_k"] / self.W[:, None]).sum(0), "h_mix": (Y * molar["h_k"] / self.W[:, None]).sum(0),
                "Wbar": Wbar, "rho": rho}
        yv = -(self.W[:, None] / Wbar) * D * gradX
        Vc = -yv.sum(1)
        j = rho * (yv + Y * Vc[:, None])
        return {**molar, **mass}, (j, Vc, (RU * cp / self.W[:, None] * j).sum(1))


def _cut(x, a, b):
    return x[..., a:b]


def _join(parts):
    """Chunks of the same nested outputs, joined along the points."""
    first = parts[0]
    if isinstance(first, torch.Tensor):
        return torch.cat(parts, dim=-1)
    if isinstance(first, dict):
        return {k: _join([p[k] for p in parts]) for k in first}
    return type(first)(_join([p[i] for p in parts]) for i in range(len(first)))


def exact(case, seed):
    path, n, K, R = case["path"], case["n"], case["K"], case["R"]
    if path == "reactor":
        return None                      # the step's solution is defined to the solver's tolerance only
    P = _Plain(_mechanism(case))
    T, p, Y = _flame(case, seed)
    extra = []
    if path in ("jvp", "train"):
        extra = list(_direction(case, seed, 0))
    if path in ("stage", "stage_f32"):
        extra = [x for j in range(DIRECTIONS) for x in _direction(case, seed, j)]
    if path == "fluxes":
        extra = [_dmix(case, seed), _grad_x(case, seed)]
    A = _dlnA(case, seed) if path == "train" else None
    gA = torch.zeros(R, dtype=torch.float64, device="cuda")
    step = max(256, int(4e7 / max(R, K * 8)))
    parts = []
    for a in range(0, n, step):
        b = min(n, a + step)
        t, q, y, *e = [_cut(x, a, b) for x in (T, p, Y, *extra)]
        if path == "rates":
            parts.append(P.rates(t, q, y))
        elif path == "transport":
            parts.append(P.transport(t, q, y))
        elif path in ("forward", "host"):
            r, tr = P.rates(t, q, y), P.transport(t, q, y)
            parts.append((r, tr) if path == "forward" else (*r, *tr))
        elif path == "jvp":
            parts.append(torch.func.jvp(lambda t_, y_: P.rates(t_, q, y_), (t, y), tuple(e))[1])
        elif path in ("stage", "stage_f32"):
            f = (lambda t_, y_: P.rates(t_, q, y_)) if path == "stage" else (lambda t_, y_: P.sources(t_, q, y_))
            jv = [torch.func.jvp(f, (t, y), (e[2 * j], e[2 * j + 1])) for j in range(DIRECTIONS)]
            parts.append((*jv[0][0], [v[1] for v in jv]))
        elif path == "train":
            tg, yg, ag = t.clone().requires_grad_(), y.clone().requires_grad_(), A.clone().requires_grad_()
            o = P.rates(tg, q, yg, ag)
            g = torch.autograd.grad(o, (tg, yg, ag), grad_outputs=(e[1], e[0]))
            gA += g[2]
            parts.append((o[0].detach(), o[1].detach(), (g[0], g[1])))
        elif path == "fluxes":
            parts.append(P.fluxes(t, q, y, *e))
    out = _join(parts)
    if path == "train":
        return out[0], out[1], (out[2][0], out[2][1], gA)
    return out
