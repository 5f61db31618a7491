"""What a program built on this framework has it do, as cases that can be timed and compared.

A ray-by-ray transport step (arXiv:1404.1719, sec. 2.1-2.2) asks, zone by zone along every ray, for
interaction rates and their Jacobian, and then solves each ray's linearised Newton system. The cases
are those calls through the package's public entry points: the pair-process rates (PairRates,
VxRatesFn), inelastic neutrino-electron scattering (NesRates), absorption and emission on nucleons
with the electron-gas closure (AbsRates, eos_eta, eos_chain) and the block-tridiagonal solve
(BlockTridiagSolver). Zone counts go from one short ray to hundreds of rays; energy grids,
quadratures, temperatures and degeneracies are those of this repository's five workloads, and the
Newton systems have the structure of its synthetic ones.

`listed` names the cases, `draw` gives more of the same ranges, `prepare` makes what a program holds
before the call, `run` is one pass, `work` what a pass cannot do without, and `exact` the same
outputs in plain 64-bit torch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1404_1719_gb300 import (AbsRates, BlockTridiagSolver, NesRates, PairRates, VxRatesFn, eos_chain,
                                   eos_eta)

RATES = ("j0", "chi0", "j1", "chi1")
SIN2W = 0.23
ETA_SWITCH = 20.0  # |eta| above which the split rule applies


# ---- the cases -------------------------------------------------------------------------------------
def _pair(name, call, rays, lo, hi, bins=21, e_max=380.0, n_mu=32, n_e=64, eta_max=20.0, radial=True,
          precision="mixed", split=False, precise=False, graph=False):
    c = dict(kind="pair", call=call, rays=rays, lo=lo, hi=hi, bins=bins, e_max=e_max, n_mu=n_mu, n_e=n_e,
             eta_max=eta_max, radial=radial, precision=precision, split=split, precise=precise, graph=graph)
    return dict(c, name=name) if name else c


def _nes(name, call, rays, lo, hi, bins=21, e_max=380.0, n_mu=16, n_e=48, eta_max=20.0, radial=True,
         precision="mixed"):
    c = dict(kind="nes", call=call, rays=rays, lo=lo, hi=hi, bins=bins, e_max=e_max, n_mu=n_mu, n_e=n_e,
             eta_max=eta_max, radial=radial, precision=precision)
    return dict(c, name=name) if name else c


def _abs(name, call, rays, lo, hi, bins=21, e_max=380.0, precision="mixed"):
    c = dict(kind="abs", call=call, rays=rays, lo=lo, hi=hi, bins=bins, e_max=e_max, eta_max=20.0, radial=True,
             precision=precision)
    return dict(c, name=name) if name else c


def _solve(name, system, rays, lo, hi, m, n_refine=2):
    c = dict(kind="solve", system=system, rays=rays, lo=lo, hi=hi, m=m, n_refine=n_refine)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: the rates of one short ray, between other parts of a program's step
        _pair("pair_rates_64_zones", "rates", 1, 64, 64, bins=17, e_max=300.0, n_mu=16, n_e=32, radial=False),
        # one ray of the paper's resolution: rates and Jacobian of a Newton iteration
        _pair("pair_newton_1_ray", "newton", 1, 400, 400),
        # the same for a node's share of the rays of a three-dimensional model
        _pair("pair_newton_128_rays", "newton", 128, 400, 400),
        # training and sensitivity runs: forward and backward through the autograd function, ragged
        # rays reaching eta_e ~ 60 under the split rule in electron energy
        _pair("pair_autograd_split", "autograd", 16, 300, 550, n_mu=16, n_e=48, eta_max=60.0, split=True),
        # the Newton blocks with respect to the partner spectra
        _pair("pair_spectral_32_rays", "spectral", 32, 400, 400),
        # the 64-bit form, for reference runs
        _pair("pair_fp64_2_rays", "rates", 2, 400, 400, precision="fp64"),
        # a host code that keeps its fields in (pinned) host memory
        _pair("pair_host_32_rays", "host", 32, 400, 400),
        # scattering: one ray, and a node's share
        _nes("nes_newton_1_ray", "newton", 1, 400, 400),
        _nes("nes_newton_64_rays", "newton", 64, 400, 400),
        # eta_e from the closure, absorption with its Jacobian, and the chain rule to (T, Y_e, rho)
        _abs("closure_absorption_512_rays", "closure", 512, 400, 400),
        # one ray's Newton system, and two rays per multiprocessor
        _solve("solve_1_ray", "newton", 1, 400, 400, 84),
        _solve("solve_304_rays", "newton", 304, 400, 400, 84),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["rates", "newton", "newton", "autograd", "spectral", "fp64", "host", "nes", "nes", "abs",
                       "solve", "solve", "solve"])
    lo = rng.choice([64, 300, 400, 400])
    hi = {64: 64, 300: 550, 400: 400}[lo]
    mean = (lo + hi) // 2
    rays = lambda zones: max(1, _log_int(rng, 1, max(1, zones // mean)))  # noqa: E731
    bins = rng.choice([13, 17, 21, 21, 25])
    e_max = rng.choice([250.0, 300.0, 380.0])
    if what == "solve":
        system = rng.choice(["newton", "newton", "dense"])
        m = rng.choice([34, 42, 50, 68, 84, 84]) if system == "newton" else rng.randint(8, 96)
        most = int(304 * 400 * 84 ** 2 / m ** 2)  # blocks no larger than those of the largest listed case
        n = min(rays(most), 304 if lo == hi else 152)
        return _solve(None, system, n, lo, hi, m, rng.choice([1, 2, 2, 2]))
    if what == "nes":
        n_mu, n_e = rng.choice([(16, 48), (16, 48), (8, 24), (12, 36)])
        if rng.random() < 0.2:
            return _nes(None, "rates", rays(800), lo, hi, bins, e_max, n_mu, n_e, 20.0, True, "fp64")
        return _nes(None, rng.choice(["rates", "newton"]), rays(25600), lo, hi, bins, e_max, n_mu, n_e,
                    rng.choice([20.0, 60.0]), rng.random() < 0.8)
    if what == "abs":
        return _abs(None, rng.choice(["rates", "closure"]), rays(204800), lo, hi, bins, e_max,
                    rng.choice(["mixed", "mixed", "mixed", "fp64"]))
    n_mu, n_e = rng.choice([(16, 32), (32, 64), (32, 64), (16, 48), (16, 20)])
    if what == "fp64":
        return _pair(None, "rates", rays(550), lo, hi, bins, e_max, n_mu, n_e, rng.choice([20.0, 60.0]), True, "fp64")
    zones = {"rates": 51200, "newton": 51200, "autograd": 12800, "spectral": 12800, "host": 12800}[what]
    mode = rng.choice(["standard", "standard", "split", "precise"])
    return _pair(None, what, rays(zones), lo, hi, bins, e_max, n_mu, n_e, rng.choice([20.0, 20.0, 60.0]),
                 rng.random() < 0.8, "mixed", mode == "split", mode == "precise", rng.random() < 0.3)


# ---- inputs ----------------------------------------------------------------------------------------
def _lengths(c):
    """Zones of each ray: fixed by the case, so that the work of a pass does not depend on the seed."""
    r = random.Random("%d %d %d" % (c["rays"], c["lo"], c["hi"]))
    return [r.randint(c["lo"], c["hi"]) for _ in range(c["rays"])]


def _zones(c):
    return sum(_lengths(c))


def _offsets(c):
    return np.concatenate([[0], np.cumsum(_lengths(c))]).astype(np.int32)


def _eps(c):
    return c["e_max"] ** (np.arange(c["bins"]) / (c["bins"] - 1))  # 1 MeV to e_max, logarithmic


def _uniform(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, dtype=torch.float64, device="cuda") * (hi - lo) + lo


def _fields(c, seed):
    """Zone states [Z][4] = (T, eta_e, Y_e, rho) and the spectra's moments J, H [Z][S][N]: radial
    profiles with 5 % noise (or independent draws), Fermi-Dirac spectra at the zone temperature."""
    g = torch.Generator("cuda").manual_seed(seed)
    Z = _zones(c)
    if c["radial"]:
        x = torch.cat([torch.linspace(0.0, 1.0, n, dtype=torch.float64) for n in _lengths(c)]).cuda()
        noise = _uniform(g, 0.95, 1.05, 4, Z)
        T = 30.0 ** (1.0 - x) * noise[0]
        eta = c["eta_max"] * (1.0 - x) * noise[1]
        ye = (0.3 + 0.2 * x) * noise[3]
        rho = 10.0 ** (14.0 - 5.0 * x) * noise[2]
        flux = 0.5 * x
    else:
        T = torch.exp(_uniform(g, 0.0, math.log(30.0), Z))
        eta = _uniform(g, 0.0, c["eta_max"], Z)
        ye = _uniform(g, 0.1, 0.5, Z)
        rho = torch.exp(_uniform(g, math.log(1e9), math.log(1e14), Z))
        flux = _uniform(g, 0.0, 0.5, Z)
    state = torch.stack([T, eta, ye, rho], 1).contiguous()
    if c["kind"] == "abs":
        return state, None, None
    eta_nu = _uniform(g, 0.0, 5.0, Z, 3)
    eps = torch.as_tensor(_eps(c)).cuda()
    J = torch.sigmoid(eta_nu[:, :, None] - eps / T[:, None, None])
    return state, J, flux[:, None, None] * J


def _seeds(c, seed):
    """Cotangents of the four rates [Z][S][N]."""
    g = torch.Generator("cuda").manual_seed(seed + 1000003)
    return [torch.randn(_zones(c), 3, c["bins"], generator=g, dtype=torch.float64, device="cuda") for _ in RATES]


def _newton_blocks(c, seed):
    """Per-ray systems with the structure of one implicit two-moment step: unknowns J, H of two
    species (m = 4 N) or of one (m = 2 N), absorption-like diagonal falling outwards over six decades,
    pair coupling to the partner species, radial fluxes coupling J and H of neighbouring zones."""
    g = torch.Generator("cuda").manual_seed(seed)
    Z, m = _zones(c), c["m"]
    S = 2 if m % 4 == 0 else 1
    N = m // (2 * S)
    x = torch.cat([torch.linspace(0.0, 1.0, n, dtype=torch.float64) for n in _lengths(c)]).cuda()
    kap = 10.0 ** (3.0 - 6.0 * x[:, None, None, None] + _uniform(g, -0.5, 0.5, Z, S, 2, N))
    rho = _uniform(g, 0.1, 0.9, Z)
    flux = 10.0 ** _uniform(g, -2.0, math.log10(3.0), Z)
    edd = _uniform(g, 1.0 / 3.0, 1.0, Z, S, N)
    A, B, C = (torch.zeros(Z, m, m, dtype=torch.float64, device="cuda") for _ in range(3))
    diag = torch.arange(m, device="cuda")
    B[:, diag, diag] = 1.0 + kap.reshape(Z, m)
    ii = torch.arange(N, device="cuda")
    first = torch.zeros(Z, dtype=torch.bool, device="cuda")
    first[torch.as_tensor(_offsets(c)[:-1].astype(np.int64)).cuda()] = True
    last = torch.roll(first, -1)
    fa, fc = torch.where(first, 0.0, flux), torch.where(last, 0.0, flux)
    for s in range(S):
        for q in range(2):
            w = _uniform(g, 0.0, 1.0, Z, N, N)
            w *= (rho[:, None] * kap[:, s, q])[..., None] / w.sum(-1, keepdim=True)
            r0, c0 = (2 * s + q) * N, (2 * (S - 1 - s) + q) * N
            B[:, r0:r0 + N, c0:c0 + N] -= w
        rJ, rH = 2 * s * N + ii, (2 * s + 1) * N + ii
        A[:, rJ, rH] = -fa[:, None].expand(Z, N)
        A[:, rH, rJ] = -fa[:, None] * edd[:, s]
        C[:, rJ, rH] = fc[:, None].expand(Z, N)
        C[:, rH, rJ] = fc[:, None] * edd[:, s]
    d = torch.randn(Z, m, generator=g, dtype=torch.float64, device="cuda")
    return A, B, C, d


def _dense_blocks(c, seed):
    """Dense blocks with uniform entries, the diagonal one and a half times its row's other entries."""
    g = torch.Generator("cuda").manual_seed(seed)
    Z, m = _zones(c), c["m"]
    A, B, C = (_uniform(g, -1.0, 1.0, Z, m, m) for _ in range(3))
    offs = torch.as_tensor(_offsets(c).astype(np.int64)).cuda()
    A[offs[:-1]] = 0.0
    C[offs[1:] - 1] = 0.0
    diag = torch.arange(m, device="cuda")
    B[:, diag, diag] = 0.0
    off = A.abs().sum(2) + B.abs().sum(2) + C.abs().sum(2)
    B[:, diag, diag] = torch.where(_uniform(g, 0.0, 1.0, Z, m) < 0.5, -1.0, 1.0) * (1.5 * off + 1.0)
    return A, B, C, torch.randn(Z, m, generator=g, dtype=torch.float64, device="cuda")


def _system(c, seed):
    return (_newton_blocks if c["system"] == "newton" else _dense_blocks)(c, seed)


def prepare(case, seed):
    c, st = case, {"case": case}
    if c["kind"] == "solve":
        st["blocks"] = _system(c, seed)
        st["offsets"] = torch.as_tensor(_offsets(c)).cuda()
        st["solver"] = BlockTridiagSolver(c["m"], _zones(c), c["n_refine"])
        st["x"] = torch.empty(_zones(c), c["m"], dtype=torch.float64, device="cuda")
        return st
    st["state"], st["J"], st["H"] = _fields(c, seed)
    if c["kind"] == "pair":
        st["rates"] = PairRates(_eps(c), c["n_mu"], c["n_e"], precision=c["precision"], split=c["split"],
                                precise=c["precise"], graph=c["graph"])
    elif c["kind"] == "nes":
        st["rates"] = NesRates(_eps(c), c["n_mu"], c["n_e"], precision=c["precision"])
    else:
        st["rates"] = AbsRates(_eps(c), precision=c["precision"])
    st["offsets"] = torch.as_tensor(_offsets(c)).cuda()
    Z, N = _zones(c), c["bins"]
    if c["call"] == "autograd":
        st["leaves"] = [t.requires_grad_() for t in (st["state"], st["J"], st["H"])]
        st["seeds"] = _seeds(c, seed)
    elif c["call"] == "host":  # pinned fields and result buffers, kept over the time steps
        st["host"] = [t.cpu().pin_memory() for t in (st["state"], st["J"], st["H"])]
        st["offsets"] = _offsets(c)
        st["out"] = {k: torch.empty(Z, 3, N, dtype=torch.float64, pin_memory=True) for k in RATES}
        st["jac"] = torch.empty(Z, 3, N, 4, 3, dtype=torch.float64, pin_memory=True)
    return st


# ---- one pass --------------------------------------------------------------------------------------
def run(st):
    c = st["case"]
    if c["kind"] == "solve":
        return st["solver"].solve(st["offsets"], *st["blocks"], out=st["x"])
    rates, call, offs = st["rates"], c["call"], st["offsets"]
    if call == "closure":
        deta = eos_eta(st["state"])
        res = rates.adjoint(st["state"], forward=True, ray_offsets=offs)
        return dict(res, state=st["state"], deta=deta, jac_rho=eos_chain(res["jac"], deta))
    if call == "autograd":
        out = VxRatesFn.apply(rates, *st["leaves"])
        grads = torch.autograd.grad(out, st["leaves"], st["seeds"])
        return dict(zip(RATES, out), state=grads[0], J=grads[1], H=grads[2])
    if call == "host":
        return rates.adjoint_host(*st["host"], ray_offsets=offs, out=st["out"], jac=st["jac"])
    if call == "spectral":
        return rates.spectral(st["state"], st["J"], st["H"], forward=True, ray_offsets=offs)
    if call == "newton":
        return rates.adjoint(st["state"], st["J"], st["H"], forward=True, ray_offsets=offs)
    return rates.evaluate(st["state"], st["J"], st["H"], ray_offsets=offs)


# ---- what a pass cannot do without -----------------------------------------------------------------
def work(case):
    """Bytes: each input read and each output written once. Flops (FMA = 2; add, mul, exp, rcp = 1):
    22 per quadrature node for rates, 34 with the tangents; 4.67 m^3 per zone for the elimination."""
    c, Z = case, _zones(case)
    if c["kind"] == "solve":
        m = c["m"]
        return {"bytes": Z * (3 * m * m + 2 * m) * 8, "flops": Z * (14.0 / 3.0) * m ** 3}
    N = c["bins"]
    SN = 3 * N
    call = c["call"]
    if c["kind"] == "abs":
        per = 4 + 4 * SN + (0 if call == "rates" else 2 * 12 * SN + 3 + 1)
        return {"bytes": 8 * Z * per, "flops": Z * SN * (20 if call == "rates" else 60)}
    nodes = Z * (N * (N + 1) // 2) * c["n_mu"] * c["n_e"]
    if c["kind"] == "nes":
        nodes = nodes * 2 // 3  # panels below the lowest electron energy hold none
    per = 4 + 2 * SN + 4 * SN
    flops = 22 * nodes
    if call in ("newton", "host"):
        per += 12 * SN
        flops = 34 * nodes
    elif call == "spectral":
        per += 12 * N * N
    elif call == "autograd":
        per += 4 * SN + 4 + 2 * SN
        flops = (22 + 34) * nodes
    return {"bytes": 8 * Z * per, "flops": flops}


# ---- the same in plain 64-bit torch ----------------------------------------------------------------
def _t(x):
    return torch.as_tensor(np.array(x, dtype=np.float64)).cuda()


def _energy_weights(eps):
    mid = np.sqrt(eps[1:] * eps[:-1])
    lo = np.concatenate([[eps[0] * math.sqrt(eps[0] / eps[1])], mid])
    hi = np.concatenate([mid, [eps[-1] * math.sqrt(eps[-1] / eps[-2])]])
    return eps ** 2 * (hi - lo)


def _couplings(species):
    cv, ca = (0.5 + 2.0 * SIN2W, 0.5) if species < 2 else (-0.5 + 2.0 * SIN2W, -0.5)
    b = ((cv + ca) ** 2, (cv - ca) ** 2)
    return b[::-1] if species == 1 else b


def _pair_kernel(c, T, eta, want_d):
    """Phi_l of term I, [z][dir][l][i][j] (dir 0 production, 1 annihilation), and its T and eta
    derivatives [z][dir][l][i][j][2]."""
    eps, N = _eps(c), c["bins"]
    i, j = np.triu_indices(N)
    t, wt = np.polynomial.legendre.leggauss(c["n_mu"])
    x, wx = np.polynomial.legendre.leggauss(c["n_e"])
    a, b, y = eps[i][:, None], eps[j][:, None], (1.0 - t)[None]
    q0, s = a + b, 2.0 * a * b * y
    q = np.sqrt(q0 * q0 - s)
    kq, kpq = a * (q0 - b * y), b * (q0 - a * y)
    perp = (a * b) ** 2 * y * (2.0 - y) / q ** 2
    pref = wt[None] * 2.0 * math.pi / (4.0 * q * a * b)
    q0, s, q, a, b, kq, kpq, perp, pref = (_t(np.broadcast_to(v, q.shape)) for v in (q0, s, q, a, b, kq, kpq, perp, pref))
    half, Em = 0.5 * q, s / (2.0 * (q0 + q))
    Tz, ez = T[:, None, None, None], eta[:, None, None, None]
    E = (Em + half)[..., None] + half[..., None] * _t(x)  # [p][m][k]
    W = half[..., None] * _t(wx)
    if c["split"]:
        xh, wh = np.polynomial.legendre.leggauss(c["n_e"] // 2)
        edge = Tz * ez
        inside = (ez > ETA_SWITCH) & (Em[..., None] < edge) & (edge < (Em + q)[..., None])
        hA, hB = 0.5 * (edge - Em[..., None]), 0.5 * ((Em + q)[..., None] - edge)
        E2 = torch.cat([edge - hA * (1.0 - _t(xh)), edge + hB * (1.0 + _t(xh))], -1)
        W2 = torch.cat([hA * _t(wh), hB * _t(wh)], -1)
        E, W = torch.where(inside, E2, E), torch.where(inside, W2, W)
    k = lambda v: v[..., None]  # noqa: E731
    Ec = (2.0 * k(q0) * E - k(s)) / (2.0 * k(q))
    pk, pkp = E * k(a) - Ec * k(kq / q), E * k(b) - Ec * k(kpq / q)
    common = pkp * pk - 0.5 * (E * E - Ec * Ec) * k(perp)
    M = [W * (v * k(0.5 * s) - common) for v in (pkp, pk)]  # terms I and II
    Eb = k(q0) - E
    fe, fp = torch.sigmoid(ez - E / Tz), torch.sigmoid(-ez - Eb / Tz)
    Oa = torch.sigmoid(E / Tz - ez) * torch.sigmoid(Eb / Tz + ez)
    f = [Oa]
    if want_d:
        f += [-Oa * (fe * E + fp * Eb) / Tz ** 2, Oa * ((1.0 - fe) * E + (1.0 - fp) * Eb) / Tz ** 2, Oa * (fp - fe)]
    boltz = torch.exp(-(_t(eps)[:, None] + _t(eps)) / T[:, None, None])
    P = torch.stack([torch.ones_like(_t(t)), _t(t)])
    ii, jj = _t(i).long(), _t(j).long()
    mats = []
    for v in f:
        full = T.new_zeros(len(T), 2, N, N)
        for X, m in enumerate(M):
            K = torch.einsum("zpmk,zpmk->zpm" if m.dim() == 4 else "zpmk,pmk->zpm", v, m) * pref
            phi = torch.einsum("zpm,lm->zlp", K, P)
            full[:, :, ii, jj] = phi if X == 0 else full[:, :, ii, jj]
            if X == 1:
                off = ii != jj
                full[:, :, jj[off], ii[off]] = phi[:, :, off]
        mats.append(full)
    phi = torch.stack([boltz[:, None] * mats[0], mats[0]], 1)
    if not want_d:
        return phi, None
    dphi = torch.stack([torch.stack([boltz[:, None] * mats[2], boltz[:, None] * mats[3]], -1),
                        torch.stack([mats[1], mats[3]], -1)], 1)
    return phi, dphi


def _nes_kernel(c, T, eta, want_d):
    """Phi_l of terms I and II, [X][z][dir][l][i][j] (dir 0 in, 1 out), and derivatives [..][2]."""
    eps, N, n_p = _eps(c), c["bins"], c["n_e"] // 3
    i, j = np.tril_indices(N)  # the down-scattering order eps_i >= eps_j
    t, wt = np.polynomial.legendre.leggauss(c["n_mu"])
    xg, wg = np.polynomial.legendre.leggauss(n_p)
    xl, wl = np.polynomial.laguerre.laggauss(n_p)
    a, b, cw = eps[i][:, None], eps[j][:, None], t[None]
    y, q0 = 1.0 - cw, a - b
    Q2 = a * a + b * b - 2.0 * a * b * cw
    Q = np.sqrt(Q2)
    kk = a * b * y
    kq, kpq = a * (a - b * cw), b * (a * cw - b)
    perp = (a * b) ** 2 * y * (2.0 - y) / Q2
    pref = wt[None] * 2.0 * math.pi / (4.0 * Q * a * b)
    a, b, q0, Q, kk, kq, kpq, perp, pref = (_t(np.broadcast_to(v, Q.shape)) for v in (a, b, q0, Q, kk, kq, kpq, perp, pref))
    Tz, ez = T[:, None, None], eta[:, None, None]
    Emin = kk / (Q + q0)
    mu = Tz * ez
    hi = torch.maximum(mu.expand(-1, *Emin.shape), Emin)
    lo = torch.maximum(mu - q0, Emin)
    bot = torch.maximum(lo - 30.0 * Tz, Emin)
    k = lambda v: v[..., None]  # noqa: E731
    panel = lambda u, v: (k(0.5 * (u + v)) + k(0.5 * (v - u)) * _t(xg), k(0.5 * (v - u)) * _t(wg))  # noqa: E731
    E1, W1 = panel(bot, lo)
    E2, W2 = panel(lo, hi)
    E3, W3 = k(hi) + k(Tz) * _t(xl), k(Tz) * _t(wl * np.exp(xl))
    E = torch.cat([E1, E2, E3], -1)
    W = torch.cat([W1, W2, W3.expand(*hi.shape, n_p)], -1)
    Ec = (E * k(q0) - k(kk)) / k(Q)
    kp, kpp = E * k(a) - Ec * k(kq / Q), E * k(b) - Ec * k(kpq / Q)
    prod = kp * kpp + 0.5 * (E * E - Ec * Ec) * k(perp)
    M = [W * (prod + k(kk) * kp), W * (prod - k(kk) * kpp)]
    Tk, ek = k(Tz), k(ez)
    Ep = E + k(q0)
    fE, cE = torch.sigmoid(ek - E / Tk), torch.sigmoid(E / Tk - ek)
    fP, cP = torch.sigmoid(ek - Ep / Tk), torch.sigmoid(Ep / Tk - ek)
    F = [cE * fP, fE * cP]  # in, out
    G = [[(-fE * E + cP * Ep) / Tk ** 2, cP - fE], [(cE * E - fP * Ep) / Tk ** 2, cE - fP]]
    P = torch.stack([torch.ones_like(_t(t)), _t(t)])
    ii, jj = _t(i).long(), _t(j).long()
    off = ii != jj

    def project(fs):  # [dir] -> [z][dir][l][i][j]; the other order exchanges in and out
        full = T.new_zeros(len(T), 2, 2, N, N)
        phi = [torch.einsum("zpm,lm->zlp", v * pref, P) for v in fs]
        for d in range(2):
            full[:, d][:, :, ii, jj] = phi[d]
            full[:, d][:, :, jj[off], ii[off]] = phi[1 - d][:, :, off]
        return full

    phis, dphis = [], []
    for m in M:
        phis.append(project([(F[d] * m).sum(-1) for d in range(2)]))
        if want_d:
            dphis.append(torch.stack([project([(F[d] * m * G[d][v]).sum(-1) for d in range(2)]) for v in range(2)], -1))
    return phis, dphis


def _contract(c, phiI, phiII, dI, dII, J, H, z, res, blocks):
    """Rates (and Jacobian, spectral blocks) of the zones z from the two terms' kernels."""
    pair = c["kind"] == "pair"
    w = _t(_energy_weights(_eps(c)))
    for s in range(3):
        p = (1, 0, 2)[s] if pair else s
        bI, bII = _couplings(s)
        K = bI * phiI + bII * phiII
        Js, Hs = J[:, p], H[:, p]
        for o in range(4):
            d, l = o & 1, o >> 1
            if pair:
                v = (1.0 - Js if o == 0 else Js) if l == 0 else Hs
            else:
                v = (Js if o == 0 else 1.0 - Js) if l == 0 else Hs
            cl = 2.0 * math.pi * (3.0 if l else 1.0) * (-1.0 if l and not pair else 1.0)
            res[RATES[o]][z, s] = cl * torch.einsum("zij,zj->zi", K[:, d, l], w * v)
            if dI is not None:
                D = bI * dI[:, d, l] + bII * dII[:, d, l]
                res["jac"][z, s, :, o, :2] = cl * torch.einsum("zijv,zj->ziv", D, w * v)
            if blocks is not None:
                blocks[z, s, o] = (-cl if o == 0 else cl) * K[:, d, l] * w


def _exact_rates(c, seed):
    state, J, H = _fields(c, seed)
    Z, N, call = _zones(c), c["bins"], c["call"]
    want_d = call in ("newton", "host", "autograd")
    per = (N * (N + 1) // 2) * c["n_mu"] * c["n_e"]
    if Z * per * (1 if c["kind"] == "pair" else 3) * (2 if want_d else 1) > 5.2e10:
        return None
    res = {k: state.new_zeros(Z, 3, N) for k in RATES}
    if want_d:
        res["jac"] = state.new_zeros(Z, 3, N, 4, 3)
    blocks = state.new_zeros(Z, 3, 4, N, N) if call in ("spectral", "autograd") else None
    step = max(1, int(3e7 // per))
    for z0 in range(0, Z, step):
        z = slice(z0, min(Z, z0 + step))
        T, eta = state[z, 0], state[z, 1]
        if c["kind"] == "pair":
            phi, d = _pair_kernel(c, T, eta, want_d)
            tr = lambda v: None if v is None else v.transpose(3, 4)  # noqa: E731
            _contract(c, phi, tr(phi), d, tr(d), J[z], H[z], z, res, blocks)
        else:
            phi, d = _nes_kernel(c, T, eta, want_d)
            d = d if want_d else [None, None]
            _contract(c, phi[0], phi[1], d[0], d[1], J[z], H[z], z, res, blocks)
    if call == "spectral":
        return dict(res, blocks=blocks)
    if call != "autograd":
        return res
    g = torch.stack(_seeds(c, seed), -1)  # [Z][S][N][4]
    jac = res.pop("jac")
    res["state"] = torch.einsum("zsio,zsiov->zv", g, jac)
    res["state"] = torch.cat([res["state"], torch.zeros_like(res["state"][:, :1])], 1)
    back = torch.einsum("zsio,zsoij->zsoj", g, blocks)[:, [1, 0, 2]]  # species s reads its partner's spectrum
    return dict(res, J=back[:, :, 0] + back[:, :, 1], H=back[:, :, 2] + back[:, :, 3])


def _exact_abs(c, seed):
    state, _, _ = _fields(c, seed)
    T, eta, ye, rho = state.unbind(1)
    deta = None
    if c["call"] == "closure":  # massless electron gas: eta^3 + pi^2 eta = 3 pi^2 n (hbar c / T)^3
        rhs = 3.0 * math.pi ** 2 * (rho * ye / 1.66053906660e-24 * 1e-39) * (197.3269804 / T) ** 3
        r = 1.5 * math.sqrt(3.0) / math.pi ** 3 * rhs
        eta = 2.0 * math.pi / math.sqrt(3.0) * torch.sinh(torch.asinh(r) / 3.0)
        slope = rhs / (3.0 * eta ** 2 + math.pi ** 2)
        deta = torch.stack([-3.0 * slope / T, slope / ye, slope / rho], 1)
    eps = _t(_eps(c))
    nb = rho / 1.66053906660e-24 * 1e-39
    res = {k: state.new_zeros(len(T), 3, c["bins"]) for k in RATES}
    jac = state.new_zeros(len(T), 3, c["bins"], 4, 3)
    for s, sg in ((0, 1.0), (1, -1.0)):  # nu_e n <-> e- p and anti-nu_e p <-> e+ n
        E = eps + sg * 1.29333236
        K = (1.0 + 3.0 * 1.2754 ** 2) / math.pi * torch.where(E > 0.0, E * E, torch.zeros_like(E))
        nn, npr = nb * (1.0 - ye), nb * ye
        nin, nout = ((nn, npr) if s == 0 else (npr, nn))
        x = E / T[:, None] - sg * eta[:, None]
        f, omf = torch.sigmoid(-x), torch.sigmoid(x)
        dT, de = f * omf * E / T[:, None] ** 2, sg * f * omf
        for o, n, v, one in ((0, nout, f, 1.0), (1, nin, omf, -1.0)):
            res[RATES[o]][:, s] = K * n[:, None] * v
            jac[:, s, :, o, 0] = one * K * n[:, None] * dT
            jac[:, s, :, o, 1] = one * K * n[:, None] * de
            jac[:, s, :, o, 2] = one * sg * K * nb[:, None] * v
    if deta is None:
        return res
    dT, de, dy = jac.unbind(-1)
    q = [deta[:, v, None, None, None] for v in range(3)]
    state = torch.stack([T, eta, ye, rho], 1)
    return dict(res, jac=jac, state=state, deta=deta, jac_rho=torch.stack([dT + de * q[0], dy + de * q[1], de * q[2]], -1))


def _exact_solve(c, seed):
    """Block elimination along all rays at once, and one correction from the residual."""
    A, B, C, d = _system(c, seed)
    n = torch.as_tensor(_lengths(c))
    starts = torch.as_tensor(_offsets(c)[:-1].astype(np.int64))
    rows = [(starts[n > k] + k).cuda() for k in range(int(n.max()))]  # zone k of every ray that has one
    lu, G = [], torch.zeros_like(A)
    piv = []
    for k, at in enumerate(rows):
        D = B[at] if k == 0 else B[at] - A[at] @ G[at - 1]
        f = torch.linalg.lu_factor(D)
        lu.append(f[0])
        piv.append(f[1])
        G[at] = torch.linalg.lu_solve(*f, C[at])

    def solve(r):
        v = torch.zeros_like(r)
        for k, at in enumerate(rows):
            b = r[at] if k == 0 else r[at] - torch.einsum("zij,zj->zi", A[at], v[at - 1])
            v[at] = torch.linalg.lu_solve(lu[k], piv[k], b[..., None])[..., 0]
        for k in range(len(rows) - 2, -1, -1):
            at = rows[k + 1] - 1  # the zones that have an outer neighbour
            v[at] -= torch.einsum("zij,zj->zi", G[at], v[at + 1])
        return v

    x = solve(d)
    r = d - torch.einsum("zij,zj->zi", B, x)
    r -= torch.einsum("zij,zj->zi", A, torch.roll(x, 1, 0))  # A is zero in a ray's first zone, C in its last
    r -= torch.einsum("zij,zj->zi", C, torch.roll(x, -1, 0))
    return x + solve(r)


def exact(case, seed):
    if case["kind"] == "solve":
        return _exact_solve(case, seed)
    return _exact_abs(case, seed) if case["kind"] == "abs" else _exact_rates(case, seed)
