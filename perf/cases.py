"""The work that programs have this library do, as cases to be timed.

A case is one call sequence of a transport code at one problem size: an implicit transport step
(mixed or FP64, with the optional physics), the energy-advection step and the neutrino stress that
follow it in the operator split, the linear system by itself, and a gradient through two steps.  The
inputs follow the post-bounce profile family of the package's `problems` module, with the matter's
angular perturbations and the opacity noise drawn from the seed.

`exact` restates each of them in plain torch FP64: dense kernels, block elimination with library
inverses, the residual driven to rounding.
"""
import math

import numpy as np
import torch

from paper_1809_05608_gb300 import adjoint as A
from paper_1809_05608_gb300 import mgfld as M

KM = 1.0e5
NS = 4
C = 2.99792458e10
HC = 1.23984198e-10
NUM = 4.0 * math.pi / HC ** 3                # number density per eps^2 d eps psi
C_NES = 2.0 * math.pi / (C * HC ** 3)
M_B = 1.674927e-24
F1 = 0.75 * (3.0 / (8.0 * math.pi)) ** (1.0 / 3.0) * HC
F2 = (4.0 / 3.0 - 1.0) / (2.5 - 1.0) * F1 * (0.5 * 2.5e14 / M_B) ** (4.0 / 3.0 - 2.5)
DT = 1e-6
GRAD_STEPS = 2
GRAD_OPACITY = 1e13                          # opacities at which the heating depends on their scales
SIGN = (1.0, -1.0, 0.0, 0.0)                 # lepton number of the species
WEIGHT = (1.0, 1.0, 2.0, 2.0)                # statistical weight


def listed():
    return [
        # one spherically symmetric ray: a 1D run, or a test; launches and the chain along the zones
        {"name": "step_fp64_1x64x12", "kind": "step", "precision": "fp64", "n_ray": 1, "n_r": 64, "n_e": 12},
        # a coarse axisymmetric run on the production grid of zones and groups
        {"name": "step_mixed_32x512x20", "kind": "step", "precision": "mixed", "n_ray": 32, "n_r": 512, "n_e": 20},
        # the benchmark's launch: an axisymmetric run of 1024 rays
        {"name": "step_mixed_1024x512x20", "kind": "step", "precision": "mixed", "n_ray": 1024, "n_r": 512, "n_e": 20},
        # the same physics in plain FP64 Newton, the reference path of a run
        {"name": "step_fp64_256x512x20", "kind": "step", "precision": "fp64", "n_ray": 256, "n_r": 512, "n_e": 20},
        # a grid of nobody's choosing: odd numbers of rays, zones and groups, with a lapse
        {"name": "step_mixed_173x301x13", "kind": "step", "precision": "mixed", "n_ray": 173, "n_r": 301, "n_e": 13,
         "lapse": True},
        # rays that cross an accretion shock
        {"name": "shock_mixed_256x512x20", "kind": "step", "precision": "mixed", "n_ray": 256, "n_r": 512, "n_e": 20,
         "shock": True, "lapse": True},
        # the flux coefficients formed at the new time level
        {"name": "coef_mixed_128x512x20", "kind": "step", "precision": "mixed", "n_ray": 128, "n_r": 512, "n_e": 20,
         "coef": True},
        # the pair process with its angular correction: coupled neutrino / antineutrino systems
        {"name": "pair_mixed_256x512x20", "kind": "step", "precision": "mixed", "n_ray": 256, "n_r": 512, "n_e": 20,
         "pair": True},
        # after the hydrodynamics: the remap in energy of the benchmark's launch
        {"name": "eadv_1024x512x20", "kind": "eadv", "n_ray": 1024, "n_r": 512, "n_e": 20},
        # the force of the neutrinos on the matter and the new lapse
        {"name": "stress_256x512x20", "kind": "stress", "n_ray": 256, "n_r": 512, "n_e": 20, "lapse": True},
        # a caller with an outer iteration of its own: the Newton system, its factors, one solution
        {"name": "linear_fp64_64x512x20", "kind": "linear", "n_ray": 64, "n_r": 512, "n_e": 20},
        # the gradient of the gain-region heating through two steps
        {"name": "grad_64x512x20", "kind": "grad", "n_ray": 64, "n_r": 512, "n_e": 20},
    ]


# the most rays a kind is drawn with (at 512 zones x 20 groups), so that none costs more than the
# largest listed case
_MOST_RAYS = {"mixed": 1024, "fp64": 256, "shock": 1024, "coef": 384, "pair": 256, "eadv": 1024, "stress": 1024,
              "linear": 256, "grad": 64}


def draw(rng):
    what = rng.choice(["mixed", "mixed", "mixed", "fp64", "fp64", "shock", "coef", "pair", "eadv", "stress", "linear",
                       "grad"])
    n_e = rng.choice([8, 12, 13, 15, 16, 17, 20, 20, 20, 24])
    n_r = int(round(math.exp(rng.uniform(math.log(48), math.log(540)))))
    most = _MOST_RAYS[what] * 512 * 400 / (max(n_r, 128) * max(n_e, 12) ** 2)
    n_ray = int(round(math.exp(rng.uniform(0.0, math.log(max(2.0, min(most, 1100.0)))))))
    case = {"kind": what, "n_ray": n_ray, "n_r": n_r, "n_e": n_e}
    if what in ("mixed", "fp64", "shock", "coef", "pair"):
        case["kind"] = "step"
        case["precision"] = what if what in ("mixed", "fp64") else "mixed"
        if what in ("shock", "coef", "pair"):
            case[what] = True
    if case["kind"] in ("step", "stress") and rng.random() < 0.5:
        case["lapse"] = True
    return case


# ------------------------------------------------------------------------------------- inputs

def _perturbation(rng, n_ray):
    """Relative angular perturbation of the rays, at most 5 %: eight cosines of the polar angle."""
    th = (np.arange(n_ray) + 0.5) * np.pi / n_ray
    c = rng.standard_normal(8)
    d = sum(c[l - 1] * np.cos(l * th) for l in range(1, 9))
    return 0.05 * d / np.sum(np.abs(c))


def _flux_factor(rc, e_g):
    r_nu = 30.0 * KM * torch.sqrt(e_g / 10.0)
    return 0.02 + 0.4 * (1.0 + torch.tanh((rc[:, :, None] - r_nu) / (5.0 * KM)))


def _species(a):
    return a[:, None].expand(-1, NS, -1, -1).contiguous()


def _inputs(case, seed):
    """The matter, grid, opacities and state of a case, FP64 on the GPU."""
    R, Z, n = case["n_ray"], case["n_r"], case["n_e"]
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def dev(a):
        return torch.as_tensor(np.array(a, dtype=np.float64, order="C"), device="cuda")

    edge = np.logspace(np.log10(10 * KM), np.log10(1e4 * KM), Z + 1)
    x = 0.5 * (edge[1:] + edge[:-1]) / (10 * KM)
    d_rho, d_T, d_s = (_perturbation(rng, R)[:, None] for _ in range(3))
    e_edge = np.logspace(np.log10(2.0), np.log10(250.0), n + 1)
    rho = dev(np.maximum(3e14 * x ** -3 * (1.0 + d_rho), 1e6))
    T = dev(np.maximum(30.0 / x * (1.0 + d_T), 0.1))
    ye = dev(np.broadcast_to(0.1 + 0.4 * np.log(x) / np.log(1e3), (R, Z)))
    e_g = dev(np.sqrt(e_edge[1:] * e_edge[:-1]))
    noise = torch.exp(0.2 * torch.randn(R, Z, n, device="cuda", dtype=torch.float64, generator=gen))
    opacity = GRAD_OPACITY if case["kind"] == "grad" else 1.0
    kappa = _species(opacity * 1e-40 * rho[:, :, None] * e_g ** 2 * noise)
    p = {"r_edge": dev(np.broadcast_to(edge, (R, Z + 1))), "lapse": None, "e_edge": dev(e_edge), "rho": rho,
         "kappa_abs": kappa, "kappa_scat": kappa.clone(), "nes_coef": 1e-41 * rho, "scale": None, "u": None,
         "eta1": None, "pair_coef": None, "pair_chi": 0}
    rc = 0.5 * (p["r_edge"][:, 1:] + p["r_edge"][:, :-1])
    if case.get("lapse") or case["kind"] == "eadv":
        p["lapse"] = torch.sqrt(1.0 - 0.2 * rc[:, :1] / rc)
    if case.get("shock"):
        r_s = dev(150.0 * KM * (1.0 + d_s))
        ramp = -0.2 * (rc - (r_s - 15.0 * KM)) / (15.0 * KM)
        beta = torch.where(rc < r_s - 15.0 * KM, torch.zeros_like(rc),
                           torch.where(rc < r_s, ramp, -0.2 * (r_s / rc) ** 2))
        p["u"] = beta * C
    if case.get("pair"):
        p["pair_coef"], p["pair_chi"] = 1e-41 * rho, 1
    if case.get("shock") or case.get("pair") or case["kind"] == "eadv":
        p["eta1"] = _species(_flux_factor(rc, e_g))
    # Fermi-Dirac occupations without a chemical potential
    psi = _species(1.0 / (1.0 + torch.exp(e_g / T[:, :, None])))
    p["state"] = (psi, ye, T)
    if case["kind"] == "eadv":
        # degenerate electron neutrinos inside, and the changes that a hydrodynamics step made
        mu = torch.where(rho > 1e12, 3.0 * T, torch.zeros_like(T))
        psi[:, 0] = 1.0 / (1.0 + torch.exp((e_g - mu[:, :, None]) / T[:, :, None]))
        xe = np.log(edge / edge[0]) / np.log(edge[-1] / edge[0])
        c_g, c_r, c_a = (rng.standard_normal((R, 4, 1)) for _ in range(3))

        def smooth(c, at, amp):
            m = np.arange(1, 5)[:, None]
            return dev(amp * np.sum(c * np.sin(np.pi * m * at), axis=1) / 4.0)
        mid = 0.5 * (xe[1:] + xe[:-1])
        p["rho_np1"] = rho * (1.0 + smooth(c_g, mid, 1e-2))
        p["r_edge_np1"] = p["r_edge"] * (1.0 - smooth(c_g, xe, 1e-2) / 3.0 + smooth(c_r, xe, 3e-4))
        p["lapse_np1"] = p["lapse"] * (1.0 + smooth(c_a, mid, 1e-4))
    if case["kind"] == "stress":
        p["p"] = 1.2435e15 * (ye * rho) ** (4.0 / 3.0) + rho * T * 1.602176634e-6 / M_B
        p["m_inner"] = 4.0 * math.pi / 3.0 * p["r_edge"][:, 0] ** 3 * rho[:, 0]
    return p


def _struct(p):
    def at(f):
        return None if p[f] is None else p[f].data_ptr()
    return M.Problem(at("r_edge"), at("lapse"), at("e_edge"), at("rho"), at("kappa_abs"), at("kappa_scat"),
                     at("nes_coef"), at("scale"), M.lib().mgfld_eos_default(), DT, M.MGFLD_BC_GHOST, at("u"),
                     at("eta1"), at("pair_coef"), p["pair_chi"])


def prepare(case, seed):
    R, Z, n = case["n_ray"], case["n_r"], case["n_e"]
    p = _inputs(case, seed)
    s = {"kind": case["kind"], "dims": M.Dims(R, Z, n, NS), "p": p}
    psi, ye, T = p["state"]

    def empty(*shape, dtype=torch.float64):
        return torch.empty(*shape, dtype=dtype, device="cuda")

    if case["kind"] == "grad":
        host = {k: (v.cpu().numpy() if isinstance(v, torch.Tensor) else v) for k, v in p.items() if k != "state"}
        inp = {"problem": dict(host, dt=DT, outer_bc=M.MGFLD_BC_GHOST), "psi0": psi.cpu().numpy()}
        s["runner"] = A.AdjointRunner(inp)
        s["scale"] = torch.ones(NS, n, dtype=torch.float64, device="cuda")
        return s
    s["struct"] = _struct(p)
    if case["kind"] == "step":
        precision = M.MGFLD_MIXED if case["precision"] == "mixed" else M.MGFLD_FP64
        size = M.mgfld_workspace_bytes_pair if case.get("pair") else M.mgfld_workspace_bytes
        s["opts"] = M.step_opts(precision, tol=1e-10 if precision == M.MGFLD_MIXED else 1e-12,
                                coef_iterate=bool(case.get("coef")))
        s["ws"] = empty(size(s["dims"], precision), dtype=torch.uint8)
        s["now"] = tuple(torch.empty_like(t) for t in p["state"])
        s["report"] = {"heating": empty(R), "ledger": empty(R, 8), "ray_status": empty(R, dtype=torch.int32),
                       "status": empty(1, dtype=torch.int32)}
    elif case["kind"] == "eadv":
        s["now"] = torch.empty_like(psi)
        s["struct"] = M.eadv_problem({"r_edge_n": p["r_edge"], "r_edge_np1": p["r_edge_np1"], "rho_n": p["rho"],
                                      "rho_np1": p["rho_np1"], "lapse_n": p["lapse"], "lapse_np1": p["lapse_np1"],
                                      "e_edge": p["e_edge"], "eta1": p["eta1"]}, limit=True)
    elif case["kind"] == "stress":
        s["ws"] = empty(M.mgfld_workspace_bytes(s["dims"], M.MGFLD_FP64), dtype=torch.uint8)
        s["out"] = {"f_edge": empty(R, Z), "f_zone": empty(R, Z), "lapse": empty(R, Z)}
    elif case["kind"] == "linear":
        s["ws"] = empty(M.mgfld_workspace_bytes(s["dims"], M.MGFLD_FP64), dtype=torch.uint8)
        s["sys"] = {"diag": empty(R, NS, Z, n, n), "lower": empty(R, NS, Z, n), "upper": empty(R, NS, Z, n),
                    "rhs": empty(R, NS, Z, n)}
        s["factor"] = empty(M.mgfld_factor_bytes(s["dims"], M.MGFLD_FP64), dtype=torch.uint8)
        s["x"] = empty(R, NS, Z, n)
    return s


# --------------------------------------------------------------------------------------- runs

def _ok(rc):
    if rc != M.MGFLD_OK:
        raise M.MgfldError(rc, "perf case")


def run(s):
    p, d = s["p"], s["dims"]
    psi0, ye0, T0 = p["state"]
    if s["kind"] == "step":
        # the state before the step is kept, as by a program that repeats a step that failed
        for now, was in zip(s["now"], p["state"]):
            now.copy_(was)
        _ok(M.mgfld_step(d, s["struct"], *s["now"], s["opts"], s["ws"], s["report"]))
        psi, ye, T = s["now"]
        return {"psi": psi, "ye": ye, "T": T, **s["report"]}
    if s["kind"] == "eadv":
        s["now"].copy_(psi0)
        _ok(M.mgfld_energy_advect(d, s["struct"], s["now"]))
        return {"psi": s["now"]}
    if s["kind"] == "stress":
        _ok(M.mgfld_stress_lapse(d, s["struct"], psi0, ye0, T0, s["ws"], p["p"], p["m_inner"], **s["out"]))
        return s["out"]
    if s["kind"] == "linear":
        _ok(M.mgfld_assemble(d, s["struct"], psi0, ye0, T0, s["sys"], s["ws"]))
        _ok(M.mgfld_factor(d, s["sys"], M.MGFLD_FP64, s["factor"]))
        _ok(M.mgfld_solve(d, s["sys"], M.MGFLD_FP64, s["factor"], s["sys"]["rhs"], s["x"]))
        return {**s["sys"], "x": s["x"]}
    leaves = [t.detach().requires_grad_() for t in (s["scale"], psi0, ye0, T0)]
    J = A.heating_objective(*leaves, s["runner"], GRAD_STEPS)
    J.backward()
    g_scale, g_psi, g_ye, g_T = (t.grad for t in leaves)
    # the occupations span 300 decades, so their gradient is taken with respect to their logarithm
    return {"J": J.detach(), "scale": g_scale, "log_psi": g_psi * psi0, "ye": g_ye, "T": g_T}


def work(case):
    """Each input read and each output written once; the arithmetic of the method: the scattering
    sums at the old state, one elimination, and (a step) one residual and one substitution for each of
    the four outer iterations that these inputs take."""
    R, Z, n = case["n_ray"], case["n_r"], case["n_e"]
    el, zones = R * NS * Z * n, R * Z
    sums, elim, subst = 4 * el * n, 2 * el * n * n, 4 * el * n
    if case["kind"] == "eadv":
        return {"bytes": 8 * (3 * el + 6 * zones), "flops": 168 * el}
    if case["kind"] == "stress":
        return {"bytes": 8 * (3 * el + 9 * zones), "flops": sums + 20 * el}
    if case["kind"] == "linear":
        return {"bytes": 8 * (el * n + 7 * el + 6 * zones), "flops": sums + elim + subst}
    if case["kind"] == "grad":
        return {"bytes": 8 * (4 * el + 8 * zones), "flops": GRAD_STEPS * (8 * (sums + subst) + 2 * elim)}
    nb = 8 * (4 * el + 7 * zones)
    if case.get("shock") or case.get("pair"):
        nb += 8 * el
    if case.get("pair"):
        elim, subst, sums = 2 * elim, 2 * subst, 2 * sums
    return {"bytes": nb, "flops": 4 * (sums + subst) + elim}


# -------------------------------------------------------------------------------- plain FP64

def _e_cold(rho, ye):
    n_e, n_n = rho * ye / M_B, rho * (1.0 - ye) / M_B
    return (F1 * n_e ** (4.0 / 3.0) + F2 * n_n ** 2.5) * M_B / rho


def _mu(rho, T, ye):
    nb = rho / M_B
    return (4.0 / 3.0 * F1 * (nb * ye) ** (1.0 / 3.0) - 2.5 * F2 * (nb * (1.0 - ye)) ** 1.5
            + T * torch.log(ye / (1.0 - ye)))


def _minerbo(eta1):
    x = eta1.clamp(0.0, 1.0)
    return 1.0 / 3.0 + 2.0 * x * x / 15.0 * (3.0 - x + 3.0 * x * x)


class _Frozen:
    """Everything of one step that its old state fixes; species are axis 1, zones 2, groups 3."""

    def __init__(self, p, state, scale=None):
        psi, ye, T = state
        E_lo, E_hi = p["e_edge"][:-1], p["e_edge"][1:]
        E = torch.sqrt((E_hi ** 2 + E_hi * E_lo + E_lo ** 2) / 3.0)
        a = p["lapse"] if p["lapse"] is not None else torch.ones_like(ye)
        re = p["r_edge"]
        self.p, self.psi_n, self.ye_n, self.T_n, self.a = p, psi, ye, T, a
        self.eps = E / a[:, :, None]
        self.W = E * E * (E_hi - E_lo) / a[:, :, None] ** 3
        self.vol = 4.0 * math.pi * (re[:, 1:] ** 3 - re[:, :-1] ** 3) / 3.0
        self.pre = (a * a / self.vol)[:, None, :, None]
        self.idt = (1.0 / (a * C * DT))[:, None, :, None]
        sc = 1.0 if scale is None else scale[None, :, None, :]
        self.kab, self.ksc = p["kappa_abs"] * sc, p["kappa_scat"] * sc
        # scattering kernels: one e-folding per temperature downwards, two upwards
        gap = (self.eps[:, :, :, None] - self.eps[:, :, None, :]) / T[:, :, None, None]
        out = torch.exp(torch.where(gap >= 0.0, -gap, 2.0 * gap))
        cw = C_NES * p["nes_coef"][:, :, None] * self.W
        self.k_out, self.k_in = cw[:, :, None, :] * out, cw[:, :, None, :] * out.transpose(2, 3)
        self.rsum = self.k_out.sum(3)[:, None]
        rc = 0.5 * (re[:, 1:] + re[:, :-1])
        self.rc, self.r_last = rc, 2.0 * re[:, -1] - rc[:, -1]
        r_r = torch.cat([rc[:, 1:], self.r_last[:, None]], 1)
        a_e = 0.5 * (a + torch.cat([a[:, 1:], a[:, -1:]], 1))
        self.i3dr = (1.0 / (3.0 * (r_r - rc)))[:, None, :, None]
        self.geo = (4.0 * math.pi * re[:, 1:] ** 2 / a_e ** 2)[:, None, :, None]
        self.re = re[:, None, :, None]
        self.j = self.emissivity(ye)
        self.coefficients(psi, self.j)
        self.sh = self.shock() if p["u"] is not None else 0.0
        if p["pair_coef"] is not None:
            self.pair()

    def sums(self, k, psi):
        return torch.matmul(psi.transpose(1, 2), k.transpose(2, 3)).transpose(1, 2)

    def emissivity(self, ye):
        mu = _mu(self.p["rho"], self.T_n, ye)
        x = torch.stack([(s * mu)[:, :, None] - self.eps for s in SIGN], 1) / self.T_n[:, None, :, None]
        return self.kab * torch.exp(x.clamp(max=700.0))

    def coefficients(self, psi, j):
        """Mean free path, neutrinosphere, ghost factor and limited edge coefficients at psi."""
        kt = self.kab + j + self.ksc + self.sums(self.k_in, psi) + self.rsum - self.sums(self.k_out, psi)
        self.lam = 1.0 / kt
        re = self.re
        dtau = (re[:, :, 1:] - re[:, :, :-1]) * kt
        tau = torch.flip(torch.cumsum(torch.flip(dtau, [2]), 2), [2])      # through the zone's inner edge
        hit = (tau >= 2.0 / 3.0).detach()
        last = hit.shape[2] - 1 - torch.argmax(torch.flip(hit.to(torch.uint8), [2]), 2)[:, :, None]
        above = (tau - dtau).gather(2, last)
        outer = re[:, :, 1:].expand_as(kt).gather(2, last)
        r_nu = outer - (2.0 / 3.0 - above) * self.lam.gather(2, last)
        self.r_nu = torch.where(hit.any(2, keepdim=True), r_nu, re[:, :, :1].expand_as(r_nu))
        rI, rg = self.rc[:, -1][:, None, None, None], self.r_last[:, None, None, None]
        rn2 = 0.25 * torch.minimum(self.r_nu, rI.expand_as(self.r_nu)) ** 2
        self.ghost = (rI * rI - rn2) / (rg * rg - rn2)
        lr = torch.cat([self.lam[:, :, 1:], self.lam[:, :, -1:]], 2)
        self.lam_e = torch.sqrt(self.lam * lr)
        pr = torch.cat([psi[:, :, 1:], self.ghost * psi[:, :, -1:]], 2)
        self.F = self.limiter(psi, pr)
        self.alpha = self.lam_e * self.F * self.i3dr * self.geo

    def limiter(self, pl, pr):
        pe, x = 0.5 * (pl + pr), self.lam_e * self.i3dr * (pr - pl).abs()
        outside = self.re[:, :, 1:] > self.r_nu
        one = torch.ones_like(x)
        m2 = torch.where(outside, 1.0 - (self.r_nu / self.re[:, :, 1:]) ** 2, one)
        h = 0.5 * (1.0 + torch.sqrt(m2))
        geom = outside & (h * pe < (1.0 - h) * x) & (pe > 1e-300)
        safe = torch.where(pe > 1e-300, pe, one)
        F = torch.where(geom, h * safe / torch.where(geom, x, one), safe / (safe + x))
        F = torch.where(pe > 1e-300, F, torch.zeros_like(F))
        # its derivative with respect to an occupation of nothing overflows, and carries nothing
        return torch.where(pe > 1e-100, F, F.detach())

    def shock(self):
        p, psi = self.p, self.psi_n
        beta = (p["u"][:, 1:] - p["u"][:, :-1]) / C
        bw = beta * ((beta.abs() - 0.01) / 0.01).clamp(0.0, 1.0)
        bw = torch.cat([bw, torch.zeros_like(bw[:, :1])], 1)[:, None, :, None]
        e3 = p["e_edge"] ** 3
        zero = torch.zeros_like(psi[..., :1])

        def ediv(m):
            at = torch.cat([zero, 0.5 * (m[..., 1:] + m[..., :-1]), zero], 3)
            return (e3[1:] * at[..., 1:] - e3[:-1] * at[..., :-1]) / ((e3[1:] - e3[:-1]) / 3.0)
        eta = p["eta1"].clamp(0.0, 1.0)
        d0 = self.alpha * bw * (ediv(eta * psi) - eta * psi)
        up = ediv(_minerbo(eta) * psi)
        d1 = -bw * torch.cat([up[:, :, 1:], up[:, :, -1:]], 2)
        return d0 + self.geo * d1 - torch.cat([torch.zeros_like(d0[:, :, :1]), d0[:, :, :-1]], 2)

    def pair(self):
        p = self.p
        cw = C_NES * p["pair_coef"][:, :, None] * self.W
        ez = torch.exp(-self.eps / self.T_n[:, :, None])
        self.k_make = cw[:, :, None, :] * ez[:, :, :, None] * ez[:, :, None, :]
        eta = p["eta1"].clamp(0.0, 1.0)
        x = 1.0 - (self.r_nu / self.rc[:, None, :, None]) ** 2
        mu = (torch.sign(x) * torch.sqrt(x.abs())).clamp(min=-1.0)
        self.k_kill = []
        for q in range(NS):
            b = q ^ 1
            c1 = 1.0 - eta[:, q, :, :, None] * eta[:, b, :, None, :] / 6.0
            m, mb = mu[:, q, :, :, None], mu[:, b, :, None, :]
            c2 = (8.0 + (m * mb - 3.0) * (1.0 + m) * (1.0 + mb)) / 8.0
            self.k_kill.append(cw[:, :, None, :] * torch.minimum(c1, c2))

    def partner(self, psi):
        """(make, kill) of the pair process."""
        other = psi[:, [1, 0, 3, 2]]
        make = self.sums(self.k_make, 1.0 - other)
        kill = torch.stack([torch.matmul(k, other[:, q, :, :, None])[..., 0] for q, k in enumerate(self.k_kill)], 1)
        return make, kill

    def source(self, psi, j):
        S = (j * (1.0 - psi) - self.kab * psi + (1.0 - psi) * self.sums(self.k_in, psi)
             - psi * (self.rsum - self.sums(self.k_out, psi)))
        if self.p["pair_coef"] is not None:
            make, kill = self.partner(psi)
            S = S + (1.0 - psi) * make - psi * kill
        return S

    def flux(self, psi):
        """A psi1 / a^2 at the outer edge of each zone."""
        return -self.alpha * (torch.cat([psi[:, :, 1:], self.ghost * psi[:, :, -1:]], 2) - psi)

    def residual(self, psi, j):
        f = self.flux(psi)
        f_in = torch.cat([torch.zeros_like(f[:, :, :1]), f[:, :, :-1]], 2)
        return (psi - self.psi_n) * self.idt + self.pre * (f - f_in + self.sh) - self.source(psi, j)

    def ye_residual(self, psi, ye, j):
        ae = (j[:, :2] * (1.0 - psi[:, :2]) - self.kab[:, :2] * psi[:, :2]) * self.W[:, None]
        net = (ae[:, 0] - ae[:, 1]).sum(2)
        return (ye - self.ye_n) * self.idt[:, 0, :, 0] + NUM * M_B / self.p["rho"] * net

    def blocks(self, psi, j, moving):
        """Dense diagonal blocks and diagonal couplings; `moving`: the limiter follows psi."""
        n = psi.shape[3]
        out, inn = self.alpha, torch.zeros_like(self.alpha)
        inn[:, :, 1:] = self.alpha[:, :, :-1]
        gh = torch.zeros_like(self.alpha)
        gh[:, :, -1:] = self.ghost
        dl, dr = out, -out
        if moving:
            with torch.enable_grad():
                l = psi.detach().clone().requires_grad_()
                r = torch.cat([psi[:, :, 1:], self.ghost * psi[:, :, -1:]], 2).detach().requires_grad_()
                flux = -self.lam_e * self.limiter(l, r) * self.i3dr * self.geo * (r - l)
                dl, dr = torch.autograd.grad(flux.sum(), (l, r))
        dl_in, dr_in = torch.zeros_like(dl), torch.zeros_like(dr)
        dl_in[:, :, 1:], dr_in[:, :, 1:] = dl[:, :, :-1], dr[:, :, :-1]
        dg = (self.idt + self.pre * (dl + gh * dr - dr_in) + j + self.kab + self.sums(self.k_in, psi) + self.rsum
              - self.sums(self.k_out, psi))
        lower, upper = -self.pre * dl_in, self.pre * dr
        upper = torch.cat([upper[:, :, :-1], torch.zeros_like(upper[:, :, :1])], 2)
        D = psi[..., None] * (self.k_in - self.k_out)[:, None] - self.k_in[:, None]
        if self.p["pair_coef"] is None:
            D += torch.diag_embed(dg)
            return D, lower, upper
        make, kill = self.partner(psi)
        D += torch.diag_embed(dg + make + kill)
        R, _, Z, _ = psi.shape
        big = torch.empty(R, 2, Z, 2 * n, 2 * n, dtype=psi.dtype, device=psi.device)
        for q in range(NS):
            o, u = (q & 1) * n, (1 - (q & 1)) * n
            big[:, q >> 1, :, o:o + n, o:o + n] = D[:, q]
            big[:, q >> 1, :, o:o + n, u:u + n] = self.k_make + psi[:, q, :, :, None] * (self.k_kill[q] - self.k_make)
        return big, _to_systems(lower, 2), _to_systems(upper, 2)


def _to_systems(v, width):
    """[ray, species, zone, group] as vectors of systems of `width` species each, and back (0)."""
    if width == 1:
        return v
    R, q, Z, n = v.shape
    if width == 2:
        return v.reshape(R, 2, 2, Z, n).transpose(2, 3).reshape(R, 2, Z, 2 * n)
    return v.reshape(R, 2, Z, 2, n // 2).transpose(2, 3).reshape(R, 4, Z, n // 2)


def _factor(D, lower, upper):
    """Inverses of the eliminated blocks, top down, in the storage of D."""
    for i in range(D.shape[2]):
        B = D[:, :, i]
        if i:
            B = B - lower[:, :, i, :, None] * D[:, :, i - 1] * upper[:, :, i - 1, None, :]
        D[:, :, i] = torch.linalg.inv(B)
    return D


def _solve(inv, lower, upper, rhs):
    x = torch.empty_like(rhs)
    Z = rhs.shape[2]
    for i in range(Z):
        b = rhs[:, :, i] - (lower[:, :, i] * x[:, :, i - 1] if i else 0.0)
        x[:, :, i] = torch.matmul(inv[:, :, i], b[..., None])[..., 0]
    for i in range(Z - 2, -1, -1):
        x[:, :, i] -= torch.matmul(inv[:, :, i], (upper[:, :, i] * x[:, :, i + 1])[..., None])[..., 0]
    return x


def _step(p, state, coef=False, scale=None):
    """One implicit step: the frozen coefficients and (psi, ye, T) with the residual at rounding."""
    f = _Frozen(p, state, scale)
    psi, ye, _ = (t.clone() for t in state)
    width = 1 if p["pair_coef"] is None else 2
    j, factors, before = f.j, None, math.inf
    for it in range(40):
        if coef and it:
            f.coefficients(psi, j)
        if factors is None or coef:
            D, lower, upper = f.blocks(psi, j, coef)
            factors = _factor(D, lower, upper), lower, upper
        d = _to_systems(_solve(*factors, _to_systems(-f.residual(psi, j), width)), width if width == 1 else 0)
        psi = psi + d
        for _ in range(3):
            h = 1e-7
            G = f.ye_residual(psi, ye, j)
            slope = (f.ye_residual(psi, ye + h, f.emissivity(ye + h)) - G) / h
            ye = ye - G / slope
            j = f.emissivity(ye)
        change = float((d.abs() / psi.abs().clamp(min=1.0)).max())
        if change < 1e-15 or (change < 1e-13 and change > 0.5 * before):
            break
        before = change
    return f, psi, ye, j


def _finish(f, psi, ye, j):
    """Temperature, ledger and gain-region heating after the step."""
    p = f.p
    S = f.source(psi, j)
    w = torch.tensor(WEIGHT, dtype=psi.dtype, device=psi.device)[None, :, None]
    sgn = torch.tensor(SIGN, dtype=psi.dtype, device=psi.device)[None, :, None]
    We = (f.W * f.eps)[:, None]
    acdt = f.a * C * DT
    e_n = _e_cold(p["rho"], f.ye_n) + 1.5 * f.T_n
    e_new = e_n - acdt * NUM * M_B / p["rho"] * (w * (We * S).sum(3)).sum(1)
    T = (e_new - _e_cold(p["rho"], ye)) / 1.5
    gain = ((f.rc >= 1.0e7) & (f.rc <= 3.0e7)).to(psi.dtype)
    heating = (-gain * acdt * f.vol * NUM * (We * S).sum(3)[:, :2].sum(1)).sum(1)
    base = p["rho"] * f.vol / M_B

    def lepton(y, s):
        return (base * y + f.vol * NUM * (sgn * (f.W[:, None] * s).sum(3)).sum(1)).sum(1)

    def energy(e, s):
        return (f.a * (base * e + f.vol * NUM * (w * (We * s).sum(3)).sum(1))).sum(1)
    out = f.flux(psi)[:, :, -1]
    E_w = f.W[:, None, -1] * f.a[:, -1][:, None, None] ** 3
    E_e = E_w * f.eps[:, None, -1] * f.a[:, -1][:, None, None]
    l0, l1 = lepton(f.ye_n, f.psi_n), lepton(ye, psi)
    e0, e1 = energy(e_n, f.psi_n), energy(e_new, psi)
    ll = C * DT * NUM * (sgn[:, :, 0] * (E_w * out).sum(2)).sum(1)
    el = C * DT * NUM * (w[:, :, 0] * (E_e * out).sum(2)).sum(1)
    return T, heating, torch.stack([l0, l1, ll, l1 + ll - l0, e0, e1, el, e1 + el - e0], 1)


def _remap(p):
    """The energy-advection step: shift, parabolic remap with the energy fix, occupation limiter."""
    psi, e = p["state"][0], p["e_edge"]
    n = psi.shape[3]
    a0, a1, r0, r1 = p["lapse"], p["lapse_np1"], p["rho"], p["rho_np1"]
    R0 = 0.5 * (p["r_edge"][:, 1:] + p["r_edge"][:, :-1])
    R1 = 0.5 * (p["r_edge_np1"][:, 1:] + p["r_edge_np1"][:, :-1])
    da, dr, db = a1 / a0 - 1.0, R1 / R0 - 1.0, R0 ** 2 * r0 / (R1 ** 2 * r1) - 1.0
    eta2 = _minerbo(p["eta1"])
    at = torch.cat([eta2[..., :1], 0.5 * (eta2[..., 1:] + eta2[..., :-1]), eta2[..., -1:]], 3)

    def zone(v):
        return v[:, None, :, None]
    Ed = e * (1.0 + zone(da - dr) - zone(db - dr) * at)
    ed, et = Ed / zone(a1), e / zone(a1).expand_as(at)

    def moment(v):
        return (v[..., 1:] ** 3 - v[..., :-1] ** 3) / 3.0

    def centre(v):
        return torch.sqrt((v[..., 1:] ** 2 + v[..., 1:] * v[..., :-1] + v[..., :-1] ** 2) / 3.0)
    nd = zone(r1 * a1 ** 3 / (r0 * a0 ** 3)) * moment(e) / moment(Ed) * psi * moment(ed)
    x = ed[..., 1:] - ed[..., :-1]
    avg = nd / x

    def ghosts(v):
        return torch.cat([v[..., :1], v[..., :1], v, v[..., -1:], v[..., -1:]], 3)
    Q, X = ghosts(avg), ghosts(x)
    d = Q[..., 1:] - Q[..., :-1]
    xl, x0, xr = X[..., :-2], X[..., 1:-1], X[..., 2:]
    dn, dp = d[..., :-1], d[..., 1:]
    s = x0 / (xl + x0 + xr) * ((2 * xl + x0) / (xr + x0) * dp + (x0 + 2 * xr) / (xl + x0) * dn)
    lim = torch.minimum(s.abs(), 2.0 * torch.minimum(dp.abs(), dn.abs())) * torch.sign(s)
    m = torch.where(dp * dn > 0.0, lim, torch.zeros_like(s))              # slopes of cells 1 .. n + 2
    xl, x0, x1, x2 = X[..., :-3], X[..., 1:-2], X[..., 2:-1], X[..., 3:]  # faces 1 .. n + 1
    t = (2 * x1 * x0 / (x0 + x1)) * ((xl + x0) / (2 * x0 + x1) - (x2 + x1) / (2 * x1 + x0)) * d[..., 1:-1]
    t = t - x0 * (xl + x0) / (2 * x0 + x1) * m[..., 1:] + x1 * (x1 + x2) / (x0 + 2 * x1) * m[..., :-1]
    face = Q[..., 1:-2] + x0 / (x0 + x1) * d[..., 1:-1] + t / (xl + x0 + x1 + x2)
    face = torch.maximum(face, torch.minimum(Q[..., 1:-2], Q[..., 2:-1]))
    face = torch.minimum(face, torch.maximum(Q[..., 1:-2], Q[..., 2:-1]))
    lo, hi = face[..., :-1], face[..., 1:]
    six = 6.0 * (avg - 0.5 * (lo + hi))
    w = hi - lo
    aL = torch.where(w * w < w * six, 3.0 * avg - 2.0 * hi, lo)
    aR = torch.where(w * w < -w * six, 3.0 * avg - 2.0 * lo, hi)
    six = 6.0 * (avg - 0.5 * (aL + aR))
    g = et[..., 1:-1] - ed[..., 1:-1]
    yu, yd = (-g / x[..., :-1]).clamp(0.0, 1.0), (g / x[..., 1:]).clamp(0.0, 1.0)
    wl, w6 = (aR - aL), six
    up = (aR[..., :-1] - 0.5 * yu * (wl[..., :-1] - (1 - 2 * yu / 3) * w6[..., :-1])) * yu * x[..., :-1]
    down = (aL[..., 1:] + 0.5 * yd * (wl[..., 1:] + (1 - 2 * yd / 3) * w6[..., 1:])) * yd * x[..., 1:]
    F = torch.where(g < 0.0, up, -down)
    F = torch.cat([torch.zeros_like(F[..., :1]), F, torch.zeros_like(F[..., :1])], 3)
    div = F[..., :-1] - F[..., 1:]
    ct = centre(et)
    s2 = (div * ct).sum(3, keepdim=True)
    s1 = (nd * (centre(ed) - ct)).sum(3, keepdim=True)
    xi = torch.where(s2 != 0.0, s1 / torch.where(s2 != 0.0, s2, torch.ones_like(s2)), torch.ones_like(s2))
    new = (nd + xi * div) / moment(et)
    wt = ct * ct * (et[..., 1:] - et[..., :-1])
    for k in range(n - 2):
        c0, c1, c2 = ct[..., k], ct[..., k + 1], ct[..., k + 2]
        c_up = (c2 - c0) * wt[..., k] / ((c2 - c1) * wt[..., k + 1])
        c_dn = (c1 - c0) * wt[..., k] / ((c2 - c1) * wt[..., k + 2])
        over = torch.minimum((new[..., k] - 1.0).clamp(min=0.0), new[..., k + 2].clamp(min=0.0) / c_dn)
        new[..., k] -= over
        new[..., k + 1] += c_up * over
        new[..., k + 2] -= c_dn * over
    return new


def _stress(p):
    f = _Frozen(p, p["state"])
    psi, a, re, rho = f.psi_n, f.a, p["r_edge"], p["rho"]
    X = psi / a[:, None, :, None] ** 4
    step = torch.cat([X[:, :, 1:], f.ghost * X[:, :, -1:]], 2) - X
    E_lo, E_hi = p["e_edge"][:-1], p["e_edge"][1:]
    E = torch.sqrt((E_hi ** 2 + E_hi * E_lo + E_lo ** 2) / 3.0)
    w = torch.tensor(WEIGHT, dtype=psi.dtype, device=psi.device)[None, :, None]
    s = (w * (f.F * step * E ** 3 * (E_hi - E_lo)).sum(3)).sum(1)
    dM = rho * f.vol
    dM_e = torch.cat([0.5 * (dM[:, 1:] + dM[:, :-1]), dM[:, -1:]], 1)
    fe = -NUM / 3.0 * 1.602176634e-6 * s * 4.0 * math.pi * re[:, 1:] ** 2 / dM_e
    fz = 0.5 * (fe + torch.cat([torch.zeros_like(fe[:, :1]), fe[:, :-1]], 1))
    mass = p["m_inner"] + dM.sum(1)
    outer = torch.sqrt(1.0 - 2.0 * 6.67430e-8 * mass / (C * C * re[:, -1]))
    rho_e = 0.5 * (rho[:, 1:] + rho[:, :-1])
    x = (p["p"][:, 1:] - p["p"][:, :-1] - dM_e[:, :-1] / (4.0 * math.pi * re[:, 1:-1] ** 2) * fe[:, :-1]) / (rho_e * C * C)
    x = torch.cat([x, torch.zeros_like(x[:, :1])], 1)
    run = torch.flip(torch.cumsum(torch.flip(x, [1]), 1), [1])
    return {"f_edge": fe, "f_zone": fz, "lapse": outer[:, None] * torch.exp(run)}


def _gradient(p, scale):
    """The heating summed over the steps; its gradients with respect to the scales, Ye and T."""
    states, J = [p["state"]], 0.0
    for _ in range(GRAD_STEPS):
        f, psi, ye, j = _step(p, states[-1], scale=scale)
        T, heating, _ = _finish(f, psi, ye, j)
        J = J + heating.sum()
        states.append((psi, ye, T))
    bars = [torch.zeros_like(t) for t in states[-1]]
    g_scale = torch.zeros_like(scale)
    for s0, s1 in zip(states[-2::-1], states[:0:-1]):
        with torch.enable_grad():
            sc, old, x = (tuple(t.detach().requires_grad_() for t in v) for v in ((scale,), s0, s1[:2]))
            f = _Frozen(p, old, sc[0])
            j = f.emissivity(x[1])
            G, GY = f.residual(x[0], j), f.ye_residual(x[0], x[1], j)
            T, heating, _ = _finish(f, x[0], x[1], j)
            L = (bars[0] * x[0]).sum() + (bars[1] * x[1]).sum() + (bars[2] * T).sum() + heating.sum()
            b_psi, b_ye = torch.autograd.grad(L, x, retain_graph=True)
        with torch.no_grad():
            D, lower, upper = f.blocks(x[0].detach(), j.detach(), False)
            zero = torch.zeros_like(lower[:, :, :1])
            lowT = torch.cat([zero, upper[:, :, :-1]], 2)
            upT = torch.cat([lower[:, :, 1:], zero], 2)
            inv = _factor(D.transpose(3, 4).contiguous(), lowT, upT)
        dYY = torch.autograd.grad(GY.sum(), x[1], retain_graph=True)[0]
        muY = torch.zeros_like(b_ye)
        for _ in range(30):
            cross = torch.autograd.grad((GY * muY).sum(), x[0], retain_graph=True)[0]
            mu = _solve(inv, lowT, upT, b_psi - cross)
            new = (b_ye - torch.autograd.grad((G * mu).sum(), x[1], retain_graph=True)[0]) / dYY
            change, muY = float((new - muY).abs().max()), new
            if change <= 1e-15 * float(new.abs().max()):
                break
        L = L - (G * mu).sum() - (GY * muY).sum()
        d_sc, *bars = torch.autograd.grad(L, (sc[0],) + old)
        g_scale = g_scale + d_sc
    return {"J": J, "scale": g_scale, "log_psi": bars[0] * p["state"][0], "ye": bars[1], "T": bars[2]}


def exact(case, seed):
    p = _inputs(case, seed)
    with torch.no_grad():
        if case["kind"] == "eadv":
            return {"psi": _remap(p)}
        if case["kind"] == "stress":
            return _stress(p)
        if case["kind"] == "linear":
            f = _Frozen(p, p["state"])
            rhs = -f.residual(f.psi_n, f.j)
            D, lower, upper = f.blocks(f.psi_n, f.j, False)
            x = _solve(_factor(D.clone(), lower, upper), lower, upper, rhs)
            return {"diag": D, "lower": lower, "upper": upper, "rhs": rhs, "x": x}
        if case["kind"] == "step":
            f, psi, ye, j = _step(p, p["state"], bool(case.get("coef")))
            T, heating, ledger = _finish(f, psi, ye, j)
            return {"psi": psi, "ye": ye, "T": T, "heating": heating, "ledger": ledger, "ray_status": None,
                    "status": None}
    n = case["n_e"]
    return _gradient(p, torch.ones(NS, n, dtype=torch.float64, device="cuda"))
