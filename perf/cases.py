"""What the library's users have it do, as cases that can be timed and compared.

A case names a call of the public Python interface (`paper_0907_3768_gb300`), the shape of its
wavelength grid and grain set, a number of cells and the options of the call.  `prepare` makes what
a radiation-transfer code holds before the call (the context with its tables and the fields and
grain numbers of one grid, on the GPU), `run` is the call, `exact` the same quantities by direct
quadrature in FP64 with torch alone.

The fields are those of the repository's workloads: a dilute stellar spectrum of strength U over
seven to ten decades, attenuated in a tenth of the cells for the widest grid, and MRN-like grain
numbers times a log-normal dust density per cell.
"""
import math

import numpy as np
import torch

import paper_0907_3768_gb300 as dust

H, CL, KB = 6.62607015e-34, 299792458.0, 1.380649e-23
SIGMA_SB = 2.0 * math.pi ** 5 * KB ** 4 / (15.0 * H ** 3 * CL ** 2)
UM = 1.0e-6
AMU = 1.66053906660e-27
J_ISRF = 2.0e-6
T_MIN, T_MAX = 2.0, 3000.0

# slope of the opacity, features (centre in um, height, relative width), bulk density, mass per atom, Einstein temperature
SPECIES = (
    (1.6, ((9.7, 1.0, 0.10),), 3500.0, 24.0 * AMU, 500.0),
    (2.0, ((0.2175, 1.0, 0.05),), 2240.0, 12.0 * AMU, 900.0),
    (2.0, tuple((c, 2.0, 0.02) for c in (3.3, 6.2, 7.7, 8.6, 11.3)), 2240.0, 12.0 * AMU, 900.0),
)

#: (wavelengths, grains) of the requests that a serving mix is made of.
MIX = ((100, 48), (200, 96), (350, 96), (500, 240))


def listed():
    return [
        # One refinement patch or one ray's cells: the smallest call of the paper's Table 1, all latency.
        dict(name="patch_32", call="solve", cells=32, K=200, sizes=32, precision="bf16x3"),
        # A one-zone or test model in plain FP32: two species of eight sizes on a coarse wavelength grid.
        dict(name="tiny_fp32", call="solve", cells=1024, K=64, sizes=8, species=2, precision="fp32"),
        # A ragged sub-grid: odd numbers of cells, wavelengths and grains.
        dict(name="subgrid_20k", call="solve", cells=20011, K=187, sizes=31, precision="bf16x3"),
        # The benchmark's grid: 2^18 cells with every output.
        dict(name="grid_262k", call="solve", cells=262144, K=200, sizes=32, precision="bf16x3"),
        # The widest wavelength grid and grain set, a tenth of the cells nearly opaque.
        dict(name="wide_131k", call="solve", cells=131072, K=500, sizes=80, precision="bf16x3", opaque=True),
        # A user who wants no split products: the FP32 contraction, rows as they come (odd stride).
        dict(name="fp32_100k", call="solve", cells=100003, K=201, sizes=32, precision="fp32"),
        # Temperatures only (sublimation, chemistry): no emission, FP16 split.
        dict(name="temps_262k", call="solve", cells=262144, K=200, sizes=32, precision="fp16x3", emission=False),
        # The paper's own form of the grain numbers: fixed per unit dust mass, one mass per cell.
        dict(name="mass_131k", call="mass", cells=131072, K=350, sizes=32, precision="bf16x3"),
        # Dust that is optically thick to its own emission: the local iteration to 1e-6.
        dict(name="coupled_16k", call="coupled", cells=16384, K=200, sizes=32, precision="bf16x3"),
        # Stochastically heated small grains of one grid, 128 energy levels.
        dict(name="fluct_16k", call="fluct", cells=16384, K=200, sizes=32, levels=128, precision="bf16x3"),
        # A CPU code that hands over page-locked host arrays and wants host arrays back.
        dict(name="host_65k", call="host", cells=65536, K=200, sizes=32, precision="bf16x3"),
        # Several simulations sharing one GPU: twelve requests of mixed shapes through the server.
        dict(name="serve_mix", call="serve", cells=240000, requests=12, precision="bf16x3"),
    ]


def draw(rng):
    call = rng.choice(("solve", "solve", "solve", "solve", "temps", "mass", "host", "coupled", "fluct", "fluct", "serve"))
    prec = rng.choice(("bf16x3", "bf16x3", "fp16x3", "fp32"))
    between = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    if call == "serve":
        return dict(call="serve", cells=between(20000, 240000), requests=rng.randint(6, 12), precision=prec)
    K, sizes = between(40, 500), between(4, 80)
    case = dict(call=call, K=K, sizes=sizes, precision=prec)
    terms = 131072 * 500 * 240  # the widest listed grid's Planck terms: no drawn case has more
    if call == "fluct":
        case["K"], case["sizes"] = between(40, 300), between(8, 40)
        case["levels"] = rng.choice((32, 64, 128, 128, 256, 512))
        case["cells"] = between(32, min(16384, 16384 * 200 * 36 * 128 // (case["K"] * case["sizes"] * 2 * case["levels"])))
        case["distribution"] = rng.random() < 0.25
        return case
    if call == "coupled":
        case["cells"] = between(32, min(16384, terms // (60 * 3 * K * sizes)))
        return case
    case["opaque"] = rng.random() < 0.3
    case["cells"] = between(32, min(262144, terms // (3 * K * sizes)))
    if call == "host":
        case["cells"] = between(1024, min(65536, terms // (3 * K * sizes)))
    if call == "temps":
        case["call"], case["emission"] = "solve", False
    return case


# ------------------------------------------------------------------ inputs

def planck(lam, T):
    x = H * CL / (lam * KB * T)
    return 2.0 * H * CL * CL / lam ** 5 / np.expm1(np.minimum(x, 700.0)) * (x < 700.0)


class Model:
    """One wavelength grid and grain set, in FP64 on the host."""

    def __init__(self, K, sizes, species=3, wide=False):
        lo, hi = (0.05, 2000.0) if wide else (0.09, 1000.0)
        a_lo = 0.00035 if species == 3 else 0.003
        self.lam = lo * UM * (hi / lo) ** (np.arange(K) / (K - 1))
        self.w = self.lam * (math.log(hi / lo) / (K - 1))
        self.w[[0, -1]] *= 0.5
        a = a_lo * UM * (1.0 / a_lo) ** (np.arange(sizes) / (sizes - 1))
        self.a = np.tile(a, species)
        self.C = np.empty((species * sizes, K))
        self.atoms, self.theta, n0 = np.empty(species * sizes), np.empty(species * sizes), []
        for s, (beta, bumps, rho, mass, theta) in enumerate(SPECIES[:species]):
            shape = (self.lam / UM) ** -beta
            shape *= 1.0 + sum(h * np.exp(-((self.lam / UM - c) ** 2) / (2.0 * (r * c) ** 2)) for c, h, r in bumps)
            of = slice(s * sizes, (s + 1) * sizes)
            self.C[of] = math.pi * a[:, None] ** 2 * np.minimum(1.0, 2.0 * math.pi * a[:, None] / self.lam) * shape
            self.atoms[of] = 4.0 / 3.0 * math.pi * a ** 3 * rho / mass
            self.theta[of] = theta
            raw = a ** -2.5
            n0.append(raw / np.sum(raw * 4.0 / 3.0 * math.pi * a ** 3))
        self.n0 = np.concatenate(n0)
        self.field = J_ISRF * (0.7 * planck(self.lam, 5000.0) / (SIGMA_SB * 5000.0 ** 4 / math.pi)
                               + 0.3 * planck(self.lam, 20000.0) / (SIGMA_SB * 20000.0 ** 4 / math.pi))
        self.extinction = (self.lam / (0.55 * UM)) ** -1.3
        self.decades = (-4.0, 6.0) if wide else (-3.0, 5.0)
        self.small = np.nonzero((self.a >= 0.5e-9) & (self.a <= 10e-9))[0]

    def context(self, precision):
        return dust.Context(self.lam, self.w, self.C, T_MIN, T_MAX, 4096, precision)


def model_of(case):
    return Model(case["K"], case["sizes"], case.get("species", 3), case.get("opaque", False))


def fields(m, cells, rng, opaque, pitch):
    """J [cells, K] on the GPU, a view of rows `pitch` long, and the cells' dust densities [cells] in FP64."""
    dev = dict(dtype=torch.float64, device="cuda")
    lo, hi = m.decades
    U = 10.0 ** (lo + (hi - lo) * torch.rand(cells, generator=rng, **dev))
    rho = torch.exp(torch.randn(cells, generator=rng, **dev))
    tau = (5.0 + 45.0 * torch.rand(cells, generator=rng, **dev)) * (torch.rand(cells, generator=rng, **dev) < 0.1)
    field, ext = torch.tensor(m.field, device="cuda"), torch.tensor(m.extinction, device="cuda")
    J = torch.zeros(cells, pitch, dtype=torch.float32, device="cuda")
    for i in range(0, cells, 65536):
        of = slice(i, i + 65536)
        row = U[of, None] * field
        if opaque:
            row *= torch.exp(-tau[of, None] * ext)
        J[of, :len(m.lam)] = row
    return J[:, :len(m.lam)], rho


def rows(K, precision):
    """Row length of J: the tensor-core precisions want a multiple of four."""
    return K if precision == "fp32" else (K + 3) // 4 * 4


def numbers(m, rho):
    return (rho[:, None] * torch.tensor(m.n0, device="cuda")).float()


def requests_of(case):
    """(wavelengths, grains, cells) of a mix's requests: cells over a factor of about thirty, at `cells` in all."""
    share = [1.35 ** i for i in range(case["requests"])]
    return [MIX[(5 * i) % len(MIX)] + (max(64, int(case["cells"] * s / sum(share))),) for i, s in enumerate(share)]


def prepare(case, seed):
    rng = torch.Generator(device="cuda").manual_seed(seed)
    if case["call"] == "serve":
        models = {kg: Model(kg[0], kg[1] // 3, 3, kg[0] == 500) for kg in MIX}
        s = dict(call="serve", contexts={kg: models[kg].context(case["precision"]) for kg in MIX}, requests=[])
        for K, G, cells in requests_of(case):
            m = models[K, G]
            J, rho = fields(m, cells, rng, K == 500, rows(K, case["precision"]))
            s["requests"].append(((K, G), J, numbers(m, rho)))
        s["server"] = dust.Server(4 << 30, 32)
        return s
    m = model_of(case)
    J, rho = fields(m, case["cells"], rng, case.get("opaque", False), rows(case["K"], case["precision"]))
    s = dict(call=case["call"], context=m.context(case["precision"]), J=J, emission=case.get("emission", True))
    if case["call"] == "mass":
        s["context"].set_grain_numbers(m.n0)
        s["m"] = rho.float()
    elif case["call"] == "fluct":
        s["context"].set_fluctuating(m.small, m.atoms[m.small], m.theta[m.small], case["levels"])
        s["n"] = numbers(m, rho)[:, m.small].contiguous()
        s["P"] = case.get("distribution", False)
    else:
        s["n"] = numbers(m, rho)
    if case["call"] == "coupled":
        # the part of a cell's emission that returns to it: up to half
        f = 0.5 * torch.rand(case["cells"], 1, generator=rng, dtype=torch.float64, device="cuda")
        E = torch.zeros(J.shape[0], J.stride(0), device="cuda")
        E[:, :case["K"]] = f / (4.0 * math.pi * (s["n"].double() @ torch.tensor(m.C, device="cuda")))
        s["E"] = E[:, :case["K"]]
    if case["call"] == "host":
        pinned = lambda *shape, kind: torch.zeros(*shape, dtype=kind, pin_memory=True).numpy()  # noqa: E731
        cells, G, ld = case["cells"], len(m.a), J.stride(0)
        whole = pinned(cells, ld, kind=torch.float32)
        whole[:, :case["K"]] = J.cpu().numpy()
        n = pinned(cells, G, kind=torch.float32)
        n[...] = s["n"].cpu().numpy()
        s.update(J=whole[:, :case["K"]], n=n, T=pinned(cells, G, kind=torch.float32), L=pinned(cells, ld, kind=torch.float32),
                 resid=pinned(cells, kind=torch.float64), flags=pinned(cells, G, kind=torch.uint8), K=case["K"])
    return s


# ------------------------------------------------------------------ the calls

def run(state):
    call = state["call"]
    if call == "serve":
        server, tickets, outs = state["server"], [], []
        for kg, J, n in state["requests"]:
            ticket, out = state["contexts"][kg].submit(server, J, n)
            tickets.append(ticket)
            outs.append(outputs(out))
        for ticket in tickets:
            server.wait(ticket)
        return outs
    ctx = state["context"]
    if call == "mass":
        return outputs(ctx.solve_mass(state["J"], state["m"]))
    if call == "coupled":
        out, iterations, change = ctx.solve_coupled(state["J"], state["E"], state["n"])
        return dict(outputs(out), iterations=iterations)
    if call == "fluct":
        out = ctx.solve_fluct(state["J"], state["n"], want_P=state["P"])
        return dict(out, L=out["L"][:, :state["J"].shape[1]])
    if call == "host":
        out = ctx.solve_host(state["J"], state["n"], state["T"], state["L"], state["resid"], state["flags"])
        return dict(out, L=out["L"][:, :state["K"]])
    if not state["emission"]:
        out = ctx.solve(state["J"], state["n"], want_L=False, want_resid=False)
        return dict(T=out["T"], flags=out["flags"])
    return outputs(ctx.solve(state["J"], state["n"]))


def outputs(out):
    return {k: out[k] for k in ("T", "L", "resid", "flags")}


def work(case):
    """Bytes: inputs and outputs once.  Flops: the contraction, and per Planck term the exponent, the
    exponential, t / (1 - t) and the weighted sum (six)."""
    if case["call"] == "serve":
        every = [solve_work(*r) for r in requests_of(case)]
        return {k: sum(w[k] for w in every) for k in ("bytes", "flops")}
    m = model_of(case)
    C, K, G = case["cells"], case["K"], len(m.a)
    if case["call"] == "fluct":
        Gf, M = len(m.small), case["levels"]
        return {"bytes": 4.0 * C * (2 * K + 2 * Gf + (Gf * M if case.get("distribution") else 0)),
                "flops": 1.0 * C * Gf * (6.0 * M * K + M * M + 4.0 * K)}
    if not case.get("emission", True):
        return {"bytes": C * (4.0 * K + 5.0 * G), "flops": 2.0 * C * K * G}
    w = solve_work(K, G, C)
    if case["call"] == "mass":
        w["bytes"] -= 4.0 * C * (G - 1)
    if case["call"] == "coupled":
        w = {"bytes": w["bytes"] + 4.0 * C * K, "flops": 20.0 * w["flops"]}  # about twenty solves to 1e-6
    return w


def solve_work(K, G, C):
    return {"bytes": C * (8.0 * K + 9.0 * G + 8.0), "flops": 8.0 * C * K * G}


# ------------------------------------------------------------------ the same in 64 bits

class Direct:
    """Eqs. 6-10 by direct quadrature in FP64 with torch, a slice of cells at a time."""

    def __init__(self, m, grains=None):
        t = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")  # noqa: E731
        self.C = t(m.C if grains is None else m.C[grains])
        self.w, self.lam = t(m.w), t(m.lam)
        self.c = H * CL / (KB * self.lam)
        self.W = self.C * self.w * (2.0 * H * CL * CL / self.lam ** 5)
        self.step = max(1, int(1.0e8 / self.W.numel()))
        self.u = torch.linspace(math.log(T_MIN), math.log(T_MAX), 2048, dtype=torch.float64, device="cuda")
        self.logP = torch.log(self.power(self.u.exp().expand(len(self.C), -1).T).T).contiguous()  # [G, nodes]

    def power(self, T):
        """sum_k w_k C[g,k] B_k(T[i,g])."""
        got = torch.empty_like(T)
        for i in range(0, len(T), self.step):
            of = slice(i, i + self.step)
            got[of] = (self.W / torch.expm1((self.c / T[of, :, None]).clamp_(max=700.0))).sum(-1)
        return got

    def temperature(self, A):
        """Roots of P_g(T) = A and their flags: the table's interpolate, then two Newton steps in ln T."""
        logA = torch.log(A)
        flags = (A < self.logP[:, 0].exp()) * 1 + (A > self.logP[:, -1].exp()) * 2
        at = torch.searchsorted(self.logP, logA.T.contiguous()).clamp_(1, len(self.u) - 1)
        y0, y1 = self.logP.gather(1, at - 1), self.logP.gather(1, at)
        u = (self.u[at - 1] + (self.u[at] - self.u[at - 1]) * ((logA.T - y0) / (y1 - y0))).T.clamp(math.log(T_MIN), math.log(T_MAX))
        for _ in range(2):
            x = (self.c / u.exp()[:, :, None]).clamp_(max=700.0)
            b = self.W / torch.expm1(x)
            P = b.sum(-1)
            u = u - (torch.log(P) - logA) * P / (b * x / -torch.expm1(-x)).sum(-1)
        T = u.exp()
        T[flags == 1], T[flags == 2] = T_MIN, T_MAX
        return T, flags.to(torch.uint8)

    def emission(self, n, T):
        L = (n[:, :, None] * (self.C / torch.expm1((self.c / T[:, :, None]).clamp_(max=700.0)))).sum(1)
        return 4.0 * math.pi * (2.0 * H * CL * CL / self.lam ** 5) * L

    def solve(self, J, n, emission=True):
        out = dict(T=[], L=[], flags=[])
        for i in range(0, len(J), self.step):
            of = slice(i, i + self.step)
            T, flags = self.temperature(J[of].double() @ (self.C * self.w).T)
            out["T"].append(T)
            out["flags"].append(flags)
            if emission:
                out["L"].append(self.emission(n[of].double(), T))
        return {k: torch.cat(v) for k, v in out.items() if v}


def exact(case, seed):
    s = prepare(case, seed)
    if case["call"] == "serve":
        direct = {kg: Direct(Model(kg[0], kg[1] // 3, 3, kg[0] == 500)) for kg in MIX}
        return [dict(direct[kg].solve(J, n), resid=None) for kg, J, n in s["requests"]]
    m = model_of(case)
    if case["call"] == "fluct":
        return distributions(m, s["J"], s["n"], case["levels"], s["P"])
    direct = Direct(m)
    if case["call"] == "host":
        got = direct.solve(torch.from_numpy(s["J"]).cuda(), torch.from_numpy(s["n"]).cuda())
        return dict({k: v.cpu().numpy() for k, v in got.items()}, resid=None)
    if case["call"] == "mass":
        return dict(direct.solve(s["J"], s["m"].double()[:, None] * torch.tensor(m.n0, device="cuda")), resid=None)
    if case["call"] == "coupled":
        J, last = s["J"].double(), None
        for _ in range(60):
            out = direct.solve(J, s["n"])
            J = s["J"].double() + s["E"].double() * out["L"]
            if last is not None and float(((out["L"] - last).abs().amax(1) / out["L"].amax(1)).max()) <= 1e-6:
                break
            last = out["L"]
        return dict(out, resid=None, iterations=None)
    if not s["emission"]:
        return direct.solve(s["J"], s["n"], emission=False)
    return dict(direct.solve(s["J"], s["n"]), resid=None)


def distributions(m, J, n, M, want_P):
    """Level populations of the fluctuating grains by the balance of the fluxes across each cut, and their emission."""
    g = m.small
    direct = Direct(m, g)
    t = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")  # noqa: E731
    theta, E0, eps = t(m.theta[g]), t(3.0 * m.atoms[g] * KB * m.theta[g]), t(H * CL / m.lam)
    lev = torch.arange(M, dtype=torch.float64, device="cuda")
    CB = direct.C * (2.0 * H * CL * CL / direct.lam ** 5)
    out = dict(L=[], dE=[], P=[])
    step = max(1, int(6.0e7 / (len(g) * M * len(m.lam))))
    for i in range(0, len(J), step):
        j = J[i:i + step].double()
        T, _ = direct.temperature(j @ (direct.C * direct.w).T)
        top = torch.minimum(2.0 * (E0 / torch.expm1(theta / T) + eps[0]), E0 / torch.expm1(theta / T_MAX))
        dE = top / (M - 1)
        Tl = theta[:, None] / torch.log1p(E0[:, None] / (dE[:, :, None] * lev[1:]))  # levels 1 .. M-1
        x = direct.c / Tl.clamp(min=T_MIN)[..., None]
        cool = (direct.W[:, None, :] / torch.expm1(x.clamp_(max=700.0))).sum(-1) / dE[:, :, None]
        R = direct.w * direct.C * j[:, None, :] / eps
        jump = (eps / dE[..., None])[:, :, None, :] - lev[1:, None] + 1.0  # a photon's levels past each jump's foot
        phi = (R[:, :, None, :] * jump.clamp_(0.0, 1.0)).sum(-1)
        P = torch.zeros(*dE.shape, M, dtype=torch.float64, device="cuda")
        P[..., 0] = 1.0
        for f in range(1, M):
            P[..., f] = (P[..., :f] * phi[..., :f].flip(-1)).sum(-1) / cool[..., f - 1]
            P /= P[..., f:f + 1].clamp(min=1.0)
        P /= P.sum(-1, keepdim=True)
        x = (direct.c / Tl[..., None]).clamp_(max=700.0)
        L = ((P[..., 1:, None] / torch.expm1(x)).sum(2) * CB * n[i:i + step].double()[:, :, None]).sum(1)
        out["L"].append(4.0 * math.pi * L)
        out["dE"].append(dE)
        out["P"].append(P)
    return {k: torch.cat(v) for k, v in out.items() if k != "P" or want_P}
