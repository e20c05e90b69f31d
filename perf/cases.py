"""Performance cases: what a user of this library has it do, through its public entry points.

A simulation case loads a state (a restart, or the next member of a study) and takes a few
steps of it; a case of the surrogate evaluates its rates, takes its gradient or fine-tunes it.
States are plume and nozzle flows of the library's own workloads with a seeded disturbance
everywhere (smooth modes in velocity, pressure, temperature and in the particle populations),
as a running flow has them, so that no cell equals its neighbour.

`exact` restates the same step in 64-bit torch, apart from the library: ideal mixture with
formation energies, MUSCL / van Leer, Roe with Harten's fix, phase change, SSP-RK2.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_2504_20742_gb300 as P
from paper_2504_20742_gb300 import surrogate as S

CFL = 0.5
FP64, FP32, FP32_MLP = P.CT_FP64, P.CT_FP32, P.CT_FP32_MLP
PRECISION = {"fp64": FP64, "fp32": FP32, "surrogate": FP32_MLP}
LAYERS = (16, 128, 128, 128, 128, 10)
MACS = sum(a * b for a, b in zip(LAYERS, LAYERS[1:]))      # of one network evaluation
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(P.__file__)), "data", "surrogate.npz")


# ---- the cases ---------------------------------------------------------------------------------
def listed():
    return [
        # the condensing quasi-1D nozzle (400 cells): the smallest grid in use, run for tens of
        # thousands of steps, so launches and latency count
        dict(name="nozzle_fp64", kind="nozzle", prec="fp64", nx=400, nr=1, steps=50),
        # a small ragged plume with freezing, as the checks against the plain method run it
        dict(name="freezing_fp64_ragged", kind="freezing", prec="fp64", nx=77, nr=29, steps=20),
        # the default workload: the kerosene plume on 1024 x 256 in FP64
        dict(name="plume_fp64", kind="kerosene", prec="fp64", nx=1024, nr=256, steps=8, tune=True),
        # a condensing plume in FP64: growth, evaporation, nucleation and freezing in over half its cells
        dict(name="mixing_fp64", kind="mixing", prec="fp64", nx=640, nr=160, steps=4, tune=True),
        # viscous and diffusive fluxes and tabulated water properties, on an odd grid
        dict(name="viscous_fp64", kind="mixing", prec="fp64", nx=501, nr=131, steps=4, viscous=True, tables=True, tune=True),
        # the large kerosene plume in FP32 (4096 x 1024, disturbed inflow rows)
        dict(name="plume_fp32", kind="kerosene", prec="fp32", nx=4096, nr=1024, steps=4, tune=True),
        # the condensing plume in FP32 (FP64 where saturation and nucleation need it)
        dict(name="mixing_fp32", kind="mixing", prec="fp32", nx=2048, nr=512, steps=4, tune=True),
        # the same with the tensor-core surrogate of the source
        dict(name="mixing_surrogate", kind="mixing", prec="surrogate", nx=1024, nr=256, steps=4, tune=True),
        # a parameter study: plumes of uneven grids and conditions in one batch
        dict(name="batch_surrogate", kind="sweep", prec="surrogate", cases=9, steps=4, tune=True),
        # an epoch of fine-tuning of the surrogate on the tensor cores, in batches of 8192
        dict(name="finetune_tc", kind="finetune", rows=131072, batch=8192, epochs=1, tensor_cores=True),
        # one FP32 gradient of a batch (a caller's own optimiser)
        dict(name="gradient_fp32", kind="gradient", rows=8192, tensor_cores=False),
        # the surrogate against the plain rates on visited states: data set and inference
        dict(name="rates_check", kind="rates", rows=200000),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("nozzle", "freezing", "kerosene", "mixing", "kerosene32", "mixing32", "mixing_mlp", "sweep", "finetune",
                       "gradient", "rates"))
    if kind == "nozzle":
        return dict(kind="nozzle", prec=rng.choice(("fp64", "fp64", "fp32")), nx=size(100, 1600), nr=1, steps=rng.randint(20, 50))
    if kind == "freezing":
        return dict(kind="freezing", prec=rng.choice(("fp64", "fp32")), nx=size(40, 300), nr=size(16, 80), steps=rng.randint(5, 20))
    if kind in ("kerosene", "mixing"):
        c = dict(kind=kind, prec="fp64", nx=size(128, 1024), nr=size(32, 256), steps=rng.randint(2, 4), tune=True)
        if kind == "mixing":
            c["nx"] = min(c["nx"], 720)
            c["nr"] = min(c["nr"], 180)
        return _options(c, rng)
    if kind == "kerosene32":
        return dict(kind="kerosene", prec="fp32", nx=size(512, 4096), nr=size(128, 1024), steps=rng.randint(2, 4), tune=True)
    if kind == "mixing32":
        return _options(dict(kind="mixing", prec="fp32", nx=size(256, 2048), nr=size(64, 512), steps=rng.randint(2, 4), tune=True), rng)
    if kind == "mixing_mlp":
        return dict(kind="mixing", prec="surrogate", nx=size(128, 1024), nr=size(32, 256), steps=rng.randint(2, 4), tune=True)
    if kind == "sweep":
        return dict(kind="sweep", prec=rng.choice(("surrogate", "fp32")), cases=rng.randint(2, 9), steps=rng.randint(2, 4), tune=True)
    if kind == "finetune":
        return dict(kind="finetune", rows=size(8192, 131072), batch=rng.choice((2048, 4096, 8192)), epochs=1, tensor_cores=rng.random() < 0.7)
    if kind == "gradient":
        return dict(kind="gradient", rows=size(500, 16384), tensor_cores=rng.random() < 0.5)
    return dict(kind="rates", rows=size(2000, 200000))


def _options(c, rng):
    """The optional parts of the model, one run in four each (the bimodal liquid alone: it has kernels of its own)."""
    if rng.random() < 0.25:
        c["bimodal"] = True
    elif rng.random() < 0.25:
        c["viscous"] = True
    if rng.random() < 0.25:
        c["tables"] = True
    return c


# ---- parameters of the flows -------------------------------------------------------------------
def _blank():
    return dict(geom=1, nx=0, nr=1, bc_xlo=0, bc_xhi=0, bc_rhi=0, phase_change=1, freezing=1, lx=1.0, lr=1.0, area_a=0.0,
                x_throat=0.0, d_core=0.0, d_fan=0.0, wall_len=0.0, T_amb=0.0, p_amb=0.0, S_ice_amb=0.0, mach_coflow=0.0,
                T_core=0.0, u_core=0.0, Yv_core=0.0, T_byp=0.0, u_byp=0.0, n_soot=0.0, soot_rm=0.0, soot_sigma=1.0, p0=0.0,
                T0=0.0, Yv_inlet=0.0, seed_l_n=0.0, seed_l_r=0.0, seed_s_n=0.0, seed_s_r=0.0, mix_width=0.0, nu_t=0.0,
                viscous=0, tables=0, equilibrium=0, bimodal=0)


def _params(case, seed):
    """The flow's parameters: those of the library's own workloads, with conditions that vary a little with the seed."""
    rs = np.random.RandomState(seed % (1 << 31))
    kind, c = case["kind"], _blank()
    c.update(nx=case.get("nx", 0), nr=case.get("nr", 1))
    if kind == "nozzle":      # 0.2 m, A/A_t = 1 + 2.5 (x/0.1 - 1)^2, moist air, no soot
        c.update(geom=0, nr=1, freezing=0, lx=0.2, area_a=2.5, x_throat=0.1, p0=40.0e3, T0=299.5 + rs.rand(), Yv_inlet=0.02)
        return c
    soot = dict(n_soot=1.0e12, soot_rm=15.0e-9, soot_sigma=1.6)
    if kind in ("kerosene", "sweep"):   # coaxial turbofan plume
        c.update(lx=32.0, lr=8.0, d_core=0.8, d_fan=2.0, T_amb=219.5 + rs.rand(), p_amb=24.0e3, S_ice_amb=1.1, mach_coflow=0.8,
                 T_core=580.0, u_core=450.0, Yv_core=0.03, T_byp=250.0, u_byp=300.0, **soot)
    else:                               # a cold moist core through a pre-mixed layer, or with a sharp edge and seeded populations
        c.update(lx=6.0, lr=2.4, d_core=0.8, d_fan=0.8, T_amb=224.5 + rs.rand(), p_amb=24.0e3, S_ice_amb=1.3, mach_coflow=0.6,
                 T_core=245.0, u_core=420.0, Yv_core=1.6e-3, T_byp=250.0, u_byp=300.0, mix_width=0.5, seed_l_n=1.0e10,
                 seed_l_r=2.0e-7, seed_s_n=1.0e8, seed_s_r=1.0e-6, **soot)
        if kind == "freezing":
            c.update(mix_width=0.0, T_core=232.0, Yv_core=4.2468e-4, u_core=250.0)
    if case.get("viscous"):
        c.update(viscous=1, nu_t=0.05)
    c.update(tables=int(bool(case.get("tables"))), bimodal=int(bool(case.get("bimodal"))))
    return c


def _sweep(case, seed):
    """A study over ambient temperature, humidity, fuel water, duct length and soot on uneven grids."""
    rs = np.random.RandomState((seed + 77) % (1 << 31))
    out = []
    for k in range(case["cases"]):
        nx = (256, 512, 1024, 2048)[(k * 7 + 3) % 4]     # the same grids for every seed
        c = _params(dict(kind="sweep", nx=nx, nr=nx // 4), seed + k)
        ei = rs.uniform(1.25, 8.9)
        lhv = 43.2 + (ei - 1.25) / (8.9 - 1.25) * (120.0 - 43.2)
        c.update(T_amb=rs.uniform(205.0, 235.0), S_ice_amb=rs.uniform(0.9, 1.3), Yv_core=0.03 * (ei / 1.25) * (43.2 / lhv),
                 wall_len=0.0 if rs.rand() < 0.5 else 1.6, n_soot=10.0 ** rs.uniform(10.0, 13.0))
        out.append(c)
    return out


def _row_factors(c, seed):
    return 1.0 + 0.01 * np.random.RandomState((seed + 1) % (1 << 31)).uniform(-1.0, 1.0, c["nr"] if c["geom"] == 1 else 1)


# ---- thermodynamics in 64 bits -------------------------------------------------------------------
RV, RA, KB, NA, MW = 8.314462618 / 0.018015, 287.05, 1.380649e-23, 6.02214076e23, 0.018015
CVA = RA / 0.4
CPA, CPV, CL, CS = CVA + RA, 1859.0, 4186.0, 2100.0
CVV = CPV - RV
E0V = 2.501e6 - (CPV - CL) * 273.15
E0S = (CL - CS) * 273.15 - 3.337e5
RHOL, RHOS, SIG_SV, PR = 1000.0, 917.0, 0.106, 0.71
FP3 = 4.0 * math.pi / 3.0
YL3, YS3 = FP3 * RHOL * 1e-18, FP3 * RHOS * 1e-18
INF = math.inf


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _lnp(T, ice):
    if ice:
        return -6024.5282 / T + 24.7219 + math.log(100.0) + 1.0613868e-2 * T - 1.3198825e-5 * T * T - 0.49382577 * torch.log(T)
    return -6096.9385 / T + 16.635794 + math.log(100.0) - 2.711193e-2 * T + 1.673952e-5 * T * T + 2.433502 * torch.log(T)


def _dlnp(T, ice):
    if ice:
        return 6024.5282 / T ** 2 + 1.0613868e-2 - 2 * 1.3198825e-5 * T - 0.49382577 / T
    return 6096.9385 / T ** 2 - 2.711193e-2 + 2 * 1.673952e-5 * T + 2.433502 / T


def _tsat(lnpv, ice):
    T = 1.0 / (1.0 / 273.15 - RV * (lnpv - math.log(611.2)) / (2.501e6 + (3.337e5 if ice else 0.0)))
    for _ in range(6):
        T = T - (_lnp(T, ice) - lnpv) / _dlnp(T, ice)
    return T


def _sigma(T):
    tau = 1.0 - T / 647.096
    return 0.2358 * tau ** 1.256 * (1.0 - 0.625 * tau)


def _cons(p, T, u, v, Yv, ml, ms, ns, mh=None):
    """Conserved fields from primitive ones (moments and soot per kg)."""
    l3 = ml[3] if mh is None else ml[3] + mh[3]
    Yl, Ys = YL3 * l3, YS3 * ms[3]
    Ya = 1.0 - Yv - Yl - Ys
    rho = p / ((Ya * RA + Yv * RV) * T)
    e = (Ya * CVA + Yv * CVV + Yl * CL + Ys * CS) * T + Yv * E0V + Ys * E0S
    f = [rho, rho * u, rho * v, rho * (e + 0.5 * (u * u + v * v)), rho * Yv] + [rho * m for m in (*ml, *ms)] + [rho * ns]
    return torch.stack(f + ([] if mh is None else [rho * m for m in mh]))


def _prim(U):
    """Primitive stencil vector (rho, u, v, p, Y_v, moments, soot per kg, ...), T, c_v, R_g."""
    rho = U[0]
    q = U / rho
    l3 = q[8] if U.shape[0] == 14 else q[8] + q[17]
    Yv, Yl, Ys = q[4], YL3 * l3, YS3 * q[12]
    Ya = 1.0 - Yv - Yl - Ys
    cv, Rg = Ya * CVA + Yv * CVV + Yl * CL + Ys * CS, Ya * RA + Yv * RV
    T = (q[3] - 0.5 * (q[1] ** 2 + q[2] ** 2) - Yv * E0V - Ys * E0S) / cv
    q = q.clone()
    q[0], q[3] = rho, rho * Rg * T
    return q, T, cv, Rg


def _vapour(pv, p):
    return pv * RA / (RV * (p - pv) + pv * RA)


def _ambient(c, dev):
    T = torch.tensor(c["T_amb"], dtype=torch.float64, device=dev)
    Yv = _vapour(c["S_ice_amb"] * torch.exp(_lnp(T, True)), c["p_amb"])
    g = ((1 - Yv) * CPA + Yv * CPV) / ((1 - Yv) * CVA + Yv * CVV)
    return T, Yv, c["mach_coflow"] * torch.sqrt(g * ((1 - Yv) * RA + Yv * RV) * T)


def _profile(c, dev):
    """T, u, Y_v and soot number per m^3 of the inflow, by row."""
    r = (torch.arange(c["nr"], dtype=torch.float64, device=dev) + 0.5) * (c["lr"] / c["nr"])
    Ta, Ya, ua = _ambient(c, dev)
    if c["mix_width"] > 0:
        w = 0.5 * (1 - torch.tanh((r - 0.5 * c["d_core"]) / c["mix_width"]))
        return w * c["T_core"] + (1 - w) * Ta, w * c["u_core"] + (1 - w) * ua, w * c["Yv_core"] + (1 - w) * Ya, w * c["n_soot"]
    core, byp = r < 0.5 * c["d_core"], r < 0.5 * c["d_fan"]

    def pick(a, b, d):
        a, b, d = (torch.as_tensor(x, dtype=torch.float64, device=dev) for x in (a, b, d))
        return torch.where(core, a, torch.where(byp, b, d))

    return pick(c["T_core"], c["T_byp"], Ta), pick(c["u_core"], c["u_byp"], ua), pick(c["Yv_core"], 0.0, Ya), pick(c["n_soot"], 0.0, 0.0)


def _gas(T, p, Yv):
    return p / (((1 - Yv) * RA + Yv * RV) * T)


def _inflow(c, ufac, dev, nf):
    """Conserved inflow rows (nf x nr) and the ambient state (nf)."""
    T, u, Yv, ns = _profile(c, dev)
    z = [torch.zeros_like(T)] * 4
    p = torch.full_like(T, c["p_amb"])
    rows = _cons(p, T, u * torch.as_tensor(ufac, device=dev), 0 * T, Yv, z, z, ns / _gas(T, p, Yv))
    Ta, Ya, ua = _ambient(c, dev)
    zero = torch.zeros_like(Ta)
    amb = _cons(zero + c["p_amb"], Ta, ua, zero, Ya, [zero] * 4, [zero] * 4, zero)
    pad = torch.zeros(nf - 14, dtype=torch.float64, device=dev)
    return torch.cat([rows, pad[:, None].expand(-1, c["nr"])]), torch.cat([amb, pad])


def _state(c, ufac, seed, dev):
    """The state a pass starts from (nf x nr x nx, float64): the inflow extended over the domain, or the isentropic
    nozzle, under seeded smooth disturbances."""
    rs = np.random.RandomState((seed + 2) % (1 << 31))
    x = (torch.arange(c["nx"], dtype=torch.float64, device=dev) + 0.5) / c["nx"]
    if c["geom"] == 0:
        g = ((1 - c["Yv_inlet"]) * CPA + c["Yv_inlet"] * CPV) / ((1 - c["Yv_inlet"]) * CVA + c["Yv_inlet"] * CVV)
        Rg = (1 - c["Yv_inlet"]) * RA + c["Yv_inlet"] * RV
        xm = x * c["lx"]
        area, sup = 1 + c["area_a"] * (xm / c["x_throat"] - 1) ** 2, xm >= c["x_throat"]
        lo, hi = torch.where(sup, 1.0, 1e-6).double(), torch.where(sup, 50.0, 1.0).double()
        for _ in range(100):
            M = 0.5 * (lo + hi)
            above = 1 / M * (2 / (g + 1) * (1 + 0.5 * (g - 1) * M * M)) ** (0.5 * (g + 1) / (g - 1)) > area
            down = above == sup
            lo, hi = torch.where(down, lo, M), torch.where(down, M, hi)
        M = 0.5 * (lo + hi)
        T = c["T0"] / (1 + 0.5 * (g - 1) * M * M)
        p = c["p0"] * (T / c["T0"]) ** (g / (g - 1))
        u = M * torch.sqrt(g * Rg * T)
        for k in range(3):
            u = u * (1 + 1e-3 * torch.cos(2 * math.pi * ((k + 1) * x + rs.rand())))
        z = [torch.zeros_like(T)] * 4
        return _cons(p, T, u, 0 * T, torch.full_like(T, c["Yv_inlet"]), z, z, 0 * T)[:, None, :].contiguous()
    r = (torch.arange(c["nr"], dtype=torch.float64, device=dev) + 0.5) / c["nr"]

    def modes(amp):
        f = torch.zeros(c["nr"], c["nx"], dtype=torch.float64, device=dev)
        for k in range(4):
            f += amp / 4 * torch.cos(2 * math.pi * ((k + 1) * r + rs.rand()))[:, None] * torch.cos(2 * math.pi * ((2 * k + 1) * x + rs.rand()))[None, :]
        return f

    T, u, Yv, ns = (a[:, None] for a in _profile(c, dev))
    uf = torch.as_tensor(ufac, device=dev)[:, None]
    T, p = T * (1 + modes(0.01)), c["p_amb"] * (1 + modes(0.005))
    u, v = u * uf * (1 + modes(0.01)), modes(4.0) * torch.sin(math.pi * r)[:, None]
    Yv, ns = Yv * (1 + modes(0.02)), ns * (1 + modes(0.05)) / _gas(T, p, Yv)
    if c["mix_width"] > 0:
        # a developed condensing plume: vapour around saturation, and water in droplets and (the
        # more the colder) in crystals, thinning out towards its edge
        plume = 0.5 * (1 - torch.tanh((r[:, None] * c["lr"] - 1.1) / 0.15)) * (1 + modes(0.3))
        plume = torch.where(plume > 0.01, plume - 0.01, 0.0)
        Yv, water, n0, cold = Yv * (1 + modes(0.4)), 4e-4 * plume, 5e11 * plume, torch.sigmoid((234 - T) / 2)

        def share(part, n, y3, sg):     # lognormal, number by kg and median radius in um
            some, ln2 = n > 0, math.log(sg) ** 2
            n = torch.where(some, n, 1.0)
            rad = (part * water / (n * y3 * math.exp(4.5 * ln2))) ** (1.0 / 3.0)
            return [torch.where(some, n * rad ** k * math.exp(0.5 * k * k * ln2), 0.0) for k in range(4)]

        ms = share(0.5 * cold, 0.05 * n0 * cold, YS3, 1.4)
        ml = share(0.2 if c["bimodal"] else 0.5, n0, YL3, 1.3)
        return _cons(p, T, u, v, Yv, ml, ms, ns, share(0.3, 0.3 * n0, YL3, 1.5) if c["bimodal"] else None).contiguous()
    core = (r * c["lr"] < 0.5 * c["d_core"])[:, None]

    def population(n, rad, sg):     # lognormal, number and median radius by kg and um
        if n <= 0:
            return [torch.zeros_like(T)] * 4
        n, rad = torch.where(core, n * (1 + modes(0.3)), 0.0), rad * 1e6 * (1 + modes(0.1))
        return [n * rad ** k * math.exp(0.5 * k * k * math.log(sg) ** 2) for k in range(4)]

    ml, ms = population(c["seed_l_n"], c["seed_l_r"], 1.3), population(c["seed_s_n"], c["seed_s_r"], 1.4)
    mh = population(0.5 * c["seed_l_n"], 2 * c["seed_l_r"], 1.3) if c["bimodal"] else None
    return _cons(p, T, u, v, Yv, ml, ms, ns, mh).contiguous()


# ---- the step in 64 bits -------------------------------------------------------------------------
def _thermo(q, het):
    Yl, Ys = YL3 * (q[8] + q[17] if het else q[8]), YS3 * q[12]
    Ya = 1 - q[4] - Yl - Ys
    cv, Rg = Ya * CVA + q[4] * CVV + Yl * CL + Ys * CS, Ya * RA + q[4] * RV
    T, ef = q[3] / (q[0] * Rg), q[4] * E0V + Ys * E0S
    return 1 + Rg / cv, (cv + Rg) * T + ef + 0.5 * (q[1] ** 2 + q[2] ** 2), ef, (1 + Rg / cv) * Rg * T


def _roe(L, R, n):
    het, t = L.shape[0] == 18, 3 - n
    (gL, HL, efL, cL), (gR, HR, efR, cR) = _thermo(L, het), _thermo(R, het)
    rt = torch.sqrt(L[0] * R[0])
    wL = L[0] / (L[0] + rt)
    wR = 1 - wL
    un, ut = wL * L[n] + wR * R[n], wL * L[t] + wR * R[t]
    H, ef, gam = wL * HL + wR * HR, wL * efL + wR * efR, 0.5 * (gL + gR)
    q2 = un * un + ut * ut
    c2 = torch.maximum((gam - 1) * (H - 0.5 * q2 - ef), 0.01 * torch.minimum(cL, cR))
    c = torch.sqrt(c2)
    dp, dun = R[3] - L[3], R[n] - L[n]
    a1, a5 = (dp - rt * c * dun) / (2 * c2), (dp + rt * c * dun) / (2 * c2)
    a2, a3 = (R[0] - L[0]) - dp / c2, rt * (R[t] - L[t])
    d = 0.1 * (un.abs() + c)
    fix = lambda l: torch.where(l < d, (l * l + d * d) / (2 * d), l)  # noqa: E731
    l1, l2, l5 = fix((un - c).abs()), un.abs(), fix((un + c).abs())
    w1, w2, w3, w5 = l1 * a1, l2 * a2, l2 * a3, l5 * a5
    mL, mR = L[0] * L[n], R[0] * R[n]
    fm = 0.5 * (mL + mR - (w1 + w2 + w5))
    F = [None] * L.shape[0]
    F[0] = fm
    F[n] = 0.5 * (mL * L[n] + L[3] + mR * R[n] + R[3] - (w1 * (un - c) + w2 * un + w5 * (un + c)))
    F[t] = 0.5 * (mL * L[t] + mR * R[t] - ((w1 + w2 + w5) * ut + w3))
    F[3] = 0.5 * (mL * HL + mR * HR - (w1 * (H - un * c) + 0.5 * w2 * q2 + w3 * ut + w5 * (H + un * c)))
    for f in range(4, L.shape[0]):
        F[f] = fm * torch.where(fm >= 0, L[f], R[f])
    return torch.stack(F)


def _transport(rho, T, p, cp, nu):
    mu = 1.716e-5 * (T / 273.15) ** 1.5 * (273.15 + 110.4) / (T + 110.4)
    return mu + rho * nu, cp * (mu / PR + rho * nu / 0.9), 2.11e-5 * (T / 273.15) ** 1.94 * 101325.0 / p + nu / 0.7, nu / 0.7


def _diffusive(a, b, ih, nu):
    def T_cp(q):
        Yl, Ys = YL3 * (q[8] + q[17] if q.shape[0] == 18 else q[8]), YS3 * q[12]
        Ya = 1 - q[4] - Yl - Ys
        return q[3] / (q[0] * (Ya * RA + q[4] * RV)), Ya * CPA + q[4] * CPV + Yl * CL + Ys * CS
    (Ta, ca), (Tb, cb) = T_cp(a), T_cp(b)
    rho, T = 0.5 * (a[0] + b[0]), 0.5 * (Ta + Tb)
    mu, lam, Dv, Dp = _transport(rho, T, 0.5 * (a[3] + b[3]), 0.5 * (ca + cb), nu)
    G = rho * Dp * ih * (b - a)
    G[0], G[1], G[2] = 0.0, mu * (b[1] - a[1]) * ih, mu * (b[2] - a[2]) * ih
    G[4] = rho * Dv * ih * (b[4] - a[4])
    ke = 0.5 * (b[1] ** 2 + b[2] ** 2 - a[1] ** 2 - a[2] ** 2)
    Gl = YL3 * (G[8] + G[17] if a.shape[0] == 18 else G[8])
    G[3] = (lam * (Tb - Ta) * ih + mu * ke * ih + ((CPV - CPA) * T + E0V) * G[4] + (CL - CPA) * T * Gl
            + ((CS - CPA) * T + E0S) * YS3 * G[12])
    return G


def _faces(q, n, dim):
    """MUSCL / van Leer states on both sides of the faces of an array with two ghost layers on each side of `dim`."""
    m = q.shape[dim]
    d = q.narrow(dim, 1, m - 1) - q.narrow(dim, 0, m - 1)
    a, b = d.narrow(dim, 0, m - 2), d.narrow(dim, 1, m - 2)
    h = torch.where(a * b > 0, a * b / torch.where(a * b > 0, a + b, 1.0), 0.0)
    mid = q.narrow(dim, 1, m - 2)
    return (mid + h).narrow(dim, 0, m - 3), (mid - h).narrow(dim, 1, m - 3)


def _ghosts(c, U, rows, amb):
    """The state with two ghost columns, and with two ghost rows, on each side."""
    nf, nr, nx = U.shape
    if c["geom"] == 0:
        u = torch.clamp(U[1, :, :1] / U[0, :, :1], min=0.0)
        Yv = torch.full_like(u, c["Yv_inlet"])
        cp = (1 - c["Yv_inlet"]) * CPA + c["Yv_inlet"] * CPV
        g = cp / ((1 - c["Yv_inlet"]) * CVA + c["Yv_inlet"] * CVV)
        T = c["T0"] - u * u / (2 * cp)
        z = [torch.zeros_like(u)] * 4
        left = _cons(c["p0"] * (T / c["T0"]) ** (g / (g - 1)), T, u, 0 * u, Yv, z, z, 0 * u)
        return torch.cat([left, left, U, U[:, :, -1:], U[:, :, -1:]], 2), None
    left = rows[:, :, None].expand(-1, -1, 2)
    flip = torch.ones(nf, 1, 1, dtype=U.dtype, device=U.device)
    flip[2] = -1.0
    top = amb[:, None, None].expand(-1, 2, nx)
    return torch.cat([left, U, U[:, :, -1:], U[:, :, -1:]], 2), torch.cat([U[:, 1:2] * flip, U[:, 0:1] * flip, U, top], 1)


def _growth(r, T, Ts, lnS, sig, rho_d, h, lam, lbar, gam, cp):
    Kn = lbar / (2 * r)
    nu = RV * Ts / h * (10.5 - 0.5 * (gam + 1) / (2 * gam) * cp * Ts / h)
    dT = Ts - T
    dTl = torch.where(lnS.abs() < 1e-8, RV * T * Ts / h, dT / torch.where(lnS.abs() < 1e-8, 1.0, lnS))
    den = rho_d * h * r * (1 + 3.78 * (1 - nu) * Kn / PR)
    return lam / den, dT - dTl * 2 * sig / (rho_d * RV * T) / r


def _slope(Ts, T, h, Yv, cv):
    a = RV * Ts * Ts / h
    return (a / Yv + (1 - a / T) * (h - RV * T) / cv).abs()


def _rates(c, q, T, cv):
    """Saturation, nucleation, growth and relaxation rates of every cell (NaN or junk where a mask says so)."""
    o, rho, Yv = {}, q[0], q[4]
    ml, ms, het = q[5:9], q[9:13], q.shape[0] == 18
    here = lambda m: (m[0] > 1e-6) & (m[1] > 0) & (m[2] > 0) & (m[3] > 0)  # noqa: E731
    o["pl"], o["ps"] = here(ml), here(ms)
    o["ph"] = here(q[14:18]) if het else torch.zeros_like(o["pl"])
    lnpv = torch.log(torch.clamp(rho * Yv * RV * T, min=1e-30))
    o["Sl"], o["Si"] = lnpv - _lnp(T, False), lnpv - _lnp(T, True)
    o["nuc"] = o["Sl"] > 0
    Yl, Ys = YL3 * (ml[3] + q[17] if het else ml[3]), YS3 * ms[3]
    Yg = 1 - Yl - Ys
    Ya = Yg - Yv
    cp = (Ya * CPA + Yv * CPV) / Yg
    gam = cp / ((Ya * CVA + Yv * CVV) / Yg)
    mu = 1.716e-5 * (T / 273.15) ** 1.5 * (273.15 + 110.4) / (T + 110.4)
    lam, lbar = mu * cp / PR, 1.5 * mu * torch.sqrt((Ya * RA + Yv * RV) / Yg * T) / q[3]
    hl, hs = (CPV - CL) * T + E0V, (CPV - CS) * T + E0V - E0S
    sig, Tl, Ti = _sigma(T), _tsat(lnpv, False), _tsat(lnpv, True)
    o["Tl"] = Tl
    # classical nucleation with the Kantrowitz factor
    S = torch.where(o["nuc"], o["Sl"], 1.0)
    rc = 2 * sig / (RHOL * RV * T * S)
    G = FP3 * sig * rc * rc / (KB * T)
    lnA = 0.5 * torch.log(2 * sig * NA ** 3 / (math.pi * MW ** 3)) + 2 * torch.log(torch.clamp(rho * Yv, min=1e-300)) - math.log(RHOL)
    soot = rho * q[13]
    gate = soot / c["n_soot"] if c["n_soot"] > 0 else 0 * soot
    o["soot"] = gate > 0
    o["lnJhom"], o["lnJhet"] = lnA - G, torch.where(o["soot"], lnA - 0.5 * G + torch.log(torch.where(o["soot"], gate, 1.0)), -INF)
    nu = RV * Tl / hl * (10.5 - 0.5 * (gam + 1) / (2 * gam) * cp * Tl / hl)
    alpha = lam / (rc * (1 + 3.78 * (1 - nu) * lbar / (2 * rc) / PR))
    o["phi"] = rho * Yv / alpha * torch.sqrt(RV * T / (2 * math.pi)) * (hl * hl / (RV * T * T) - hl / T)
    o["Jhom"], o["Jhet"] = (torch.where(o["nuc"], torch.exp(o[k]) / (1 + o["phi"]), 0.0) for k in ("lnJhom", "lnJhet"))
    o["rc"] = torch.where(o["nuc"], rc * 1e6, 0.0)

    def grow(m, ok, Ts, lnS, sg, rd, h):
        m0, m2 = torch.where(ok, m[0], 1.0), torch.where(ok, m[2], 1.0)
        cond, D = _growth(torch.sqrt(m2 / m0) * 1e-6, T, Ts, lnS, sg, rd, h, lam, lbar, gam, cp)
        return (torch.where(ok, cond * D * 1e6, 0.0), torch.where(ok, 4 * math.pi * rd * 1e-12 * m2 * cond * _slope(Ts, T, h, Yv, cv), 0.0))

    o["Gl"], o["xl"] = grow(ml, o["pl"], Tl, o["Sl"], sig, RHOL, hl)
    o["Gs"], o["xs"] = grow(ms, o["ps"], Ti, o["Si"], SIG_SV, RHOS, hs)
    o["Gh"], o["xh"] = grow(q[14:18], o["ph"], Tl, o["Sl"], sig, RHOL, hl) if het else (0 * T, 0 * T)
    o["active"] = o["nuc"] | o["pl"] | o["ps"] | o["ph"]
    return o


def _rp2(c):
    return c["soot_rm"] ** 2 * math.exp(2 * math.log(c["soot_sigma"]) ** 2)


def _features(c, q, T, o):
    ln = lambda a, lo: torch.log(torch.clamp(a, min=lo))  # noqa: E731
    x = [torch.log(q[3]), T, 1 / torch.clamp(o["Sl"], min=0.25) ** 2, ln(q[4], 1e-12)] + [ln(m, 1e-30) for m in q[5:13]]
    x += [ln(q[0] * q[13], 1.0), torch.full_like(T, math.log(_rp2(c) * 1e12 + 1e-30)), o["Sl"], o["Si"]]
    return torch.stack(x, -1)


def _weights():
    z = np.load(WEIGHTS)
    return {k: z[k] for k in z.files}


def _network(z, x, dev):
    """The packed network in 64 bits on raw inputs (rows x 16) -> raw outputs (rows x 10)."""
    t = lambda k: torch.as_tensor(z[k].astype(np.float64), device=dev)  # noqa: E731
    sd = t("x_sd")
    h, p, at = (x - t("x_mean")) / torch.where(sd > 0, sd, 1.0), t("params"), 0
    for l in range(5):
        i, n = LAYERS[l], LAYERS[l + 1]
        h = h @ p[at:at + i * n].view(n, i).T + p[at + i * n:at + i * n + n]
        h = h * torch.sigmoid(h) if l < 4 else h
        at += i * n + n
    return h * t("y_sd") + t("y_mean")


def _surrogate_rates(c, q, T, o, z):
    dev = T.device
    x = _features(c, q, T, o).reshape(-1, 16)
    lo, hi = (torch.as_tensor(z[k].astype(np.float64), device=dev) for k in ("x_min", "x_max"))
    eps = 1e-6     # the hull is in 32 bits, and one input is a constant of the case
    inside = ((x >= lo - eps * lo.abs()) & (x <= hi + eps * hi.abs())).all(1) & o["active"].reshape(-1)
    y = torch.zeros(x.shape[0], 10, dtype=torch.float64, device=dev)
    if bool(inside.any()):
        y[inside] = _network(z, x[inside], dev)
    lo, hi = (torch.as_tensor(z[k].astype(np.float64), device=dev) for k in ("y_min", "y_max"))
    y = torch.minimum(torch.maximum(y, lo), hi).reshape(*T.shape, 10)
    inside = inside.reshape(T.shape)
    for k, ok, v in (("Gl", "pl", torch.sinh(y[..., 2])), ("Gs", "ps", torch.sinh(y[..., 3])), ("xl", "pl", torch.exp(y[..., 4])),
                     ("xs", "ps", torch.exp(y[..., 5]))):
        o[k] = torch.where(inside, torch.where(o[ok], v, 0.0), o[k])


def _source(c, U, q, T, cv, acc, dt, z):
    """Phase-change rates of the conserved fields, limited on the flux-updated state."""
    rho, het = q[0], q.shape[0] == 18
    o = _rates(c, q, T, cv)
    if z is not None:
        _surrogate_rates(c, q, T, o, z)
    ml, ms = q[5:9], q[9:13]
    x = dt * (o["xl"] + o["xs"] + o["xh"])
    th = torch.where(x > 0, -torch.expm1(-x) / torch.where(x > 0, x, 1.0), 1.0)
    Gl, Gs, Gh = o["Gl"] * th, o["Gs"] * th, o["Gh"] * th
    daw = 1 - torch.exp(o["Sl"] - o["Si"])
    d = torch.clamp(daw, max=0.34)
    l10 = -906.7 + d * (8502.0 + d * (-26924.0 + d * 29180.0))
    Js = torch.where(daw >= 0.26, 10.0 ** torch.clamp(l10, max=60.0) * 1e6, 0.0)
    kimm = 1e8 * 4 * math.pi * _rp2(c)
    cold = (T < 273.15) if c["freezing"] else torch.zeros_like(o["pl"])

    def freeze(m, ok, soot):
        ok = ok & cold
        m0, m3 = torch.where(ok, m[0], 1.0), torch.where(ok, m[3], 1.0)
        rv = (m3 / m0) ** (1.0 / 3.0)
        om = Js * FP3 * (rv * 1e-6) ** 3 + (kimm * torch.clamp(q[13] / m0, max=1.0) if soot else 0.0)
        return torch.where(ok, m0 * -torch.expm1(-om * dt) / dt, 0.0), torch.where(ok, rv, 0.0)

    Nf, rv = freeze(ml, o["pl"], not het)
    Nh, rh = freeze(q[14:18], o["ph"], True) if het else (0 * T, 0 * T)
    kk, cube = range(4), (RHOL / RHOS) ** (1.0 / 3.0)
    J = (o["Jhom"] if het else o["Jhom"] + o["Jhet"]) / rho
    up = lambda m, G, k: k * m[k - 1] * G if k else 0 * T  # noqa: E731
    dl = [up(ml, Gl, k) + J * o["rc"] ** k - Nf * rv ** k for k in kk]
    ds = [up(ms, Gs, k) + Nf * (rv * cube) ** k + Nh * (rh * cube) ** k for k in kk]
    dh = [up(q[14:18], Gh, k) + o["Jhet"] / rho * o["rc"] ** k - Nh * rh ** k for k in kk] if het else []
    A = (U + dt * acc) / rho
    for dm, at in ((dl, 5), (ds, 9), (dh, 14)):
        if dm:
            gone = A[at + 3] + dt * dm[3] <= 0
            for k in kk:
                dm[k] = torch.where(gone, -A[at + k] / dt, dm[k])
    dY = -(YL3 * (dl[3] + dh[3] if het else dl[3]) + YS3 * ds[3])
    dry = A[4] + dt * dY < 0
    th = torch.where(dry, torch.where(A[4] > 0, A[4] / torch.where(dry, -dt * dY, 1.0), 0.0), 1.0)
    Q = torch.zeros_like(U)
    Q[4] = dY * th
    for k in kk:
        Q[5 + k], Q[9 + k] = dl[k] * th, ds[k] * th
        if het:
            Q[14 + k] = dh[k] * th
    return torch.where(o["active"], rho * Q, 0.0)


def _residual(c, U, rows, amb, dt, z):
    nf, nr, nx = U.shape
    dx = c["lx"] / nx
    Ux, Ur = _ghosts(c, U, rows, amb)
    q, T, cv, _ = _prim(U)
    qx = _prim(Ux)[0]
    F = _roe(*_faces(qx, 1, 2), 1)
    if c["viscous"]:
        F = F - _diffusive(qx[:, :, 1:-2], qx[:, :, 2:-1], 1 / dx, c["nu_t"])
    if c["geom"] == 0:
        area = lambda i: 1 + c["area_a"] * (i * dx / c["x_throat"] - 1) ** 2  # noqa: E731
        i = torch.arange(nx + 1, dtype=torch.float64, device=U.device)
        Af, Ac = area(i), area(i[:-1] + 0.5)
        acc = (Af[:-1] * F[:, :, :-1] - Af[1:] * F[:, :, 1:]) / (Ac * dx)
        acc[1] += q[3] * (Af[1:] - Af[:-1]) / (Ac * dx)
        return acc + _source(c, U, q, T, cv, acc, dt, z)
    dr = c["lr"] / nr
    acc = (F[:, :, :-1] - F[:, :, 1:]) / dx
    del F, qx, Ux
    qr = _prim(Ur)[0]
    F = _roe(*_faces(qr, 2, 1), 2)
    if c["viscous"]:
        F = F - _diffusive(qr[:, 1:-2], qr[:, 2:-1], 1 / dr, c["nu_t"])
    j = torch.arange(nr, dtype=torch.float64, device=U.device)[:, None]
    south, north = F[:, :-1].clone(), F[:, 1:].clone()
    jw = int(math.floor(0.5 * c["d_fan"] / dr + 0.5))
    cols = int(((np.arange(nx) + 0.5) * dx < c["wall_len"]).sum()) if c["wall_len"] > 0 else 0
    for row, side in ((jw, south), (jw - 1, north)):     # the duct wall carries the pressure only
        if cols and 0 <= row < nr:
            side[:, row, :cols] = 0.0
            side[2, row, :cols] = q[3, row, :cols]
    acc += (j * south - (j + 1) * north) / ((j + 0.5) * dr)
    acc[2] += q[3] / ((j + 0.5) * dr)
    if c["viscous"]:
        Yl, Ys = YL3 * (q[8] + q[17] if nf == 18 else q[8]), YS3 * q[12]
        cp = (1 - q[4] - Yl - Ys) * CPA + q[4] * CPV + Yl * CL + Ys * CS
        acc[2] -= _transport(q[0], T, q[3], cp, c["nu_t"])[0] * q[2] / ((j + 0.5) * dr) ** 2
    return acc + _source(c, U, q, T, cv, acc, dt, z)


def _dt(c, U):
    q, T, cv, Rg = _prim(U)
    dx, dr = c["lx"] / c["nx"], c["lr"] / c["nr"]
    a = torch.sqrt((1 + Rg / cv) * Rg * T)
    rate = (q[1].abs() + a) / dx
    if c["geom"] == 1:
        rate = rate + (q[2].abs() + a) / dr
    if c["viscous"]:
        Yl, Ys = YL3 * (q[8] + q[17] if U.shape[0] == 18 else q[8]), YS3 * q[12]
        cp = (1 - q[4] - Yl - Ys) * CPA + q[4] * CPV + Yl * CL + Ys * CS
        mu, lam, Dv, Dp = _transport(q[0], T, q[3], cp, c["nu_t"])
        nu = torch.maximum(torch.maximum(mu / q[0], lam / (q[0] * cv)), Dv)
        rate = rate + 2 * torch.clamp(nu, min=Dp) * (1 / dx ** 2 + 1 / dr ** 2)
    return CFL / rate.max()


def _advance(c, ufac, U, steps, z=None):
    U = U.double()
    rows, amb = _inflow(c, ufac, U.device, U.shape[0]) if c["geom"] == 1 else (None, None)
    for _ in range(steps):
        dt = _dt(c, U)
        U1 = U + dt * _residual(c, U, rows, amb, dt, z)
        U = 0.5 * U + 0.5 * (U1 + dt * _residual(c, U1, rows, amb, dt, z))
    return U


def _fields(U):
    """The state by what its fields are: each is compared on its own scale."""
    out = dict(rho=U[0], momentum=U[1:3], energy=U[3], vapour=U[4], liquid=U[5:9], ice=U[9:13], soot=U[13])
    if U.shape[0] == 18:
        out["liquid_het"] = U[14:18]
    return out


# ---- states and training rows of the surrogate -----------------------------------------------------
def _visited(n, seed, dev):
    """n conserved states as condensing plumes visit them (n x 14, float64)."""
    g = torch.Generator(device="cpu").manual_seed(seed)
    rnd = torch.rand(16, n, generator=g, dtype=torch.float64).to(dev)
    T, p = 205 + 70 * rnd[0], 24.0e3 * (0.6 + 0.8 * rnd[1])
    S = torch.exp(math.log(0.6) + rnd[2] * math.log(8.0 / 0.6))
    Yv = torch.clamp(_vapour(torch.minimum(S * torch.exp(_lnp(T, False)), 0.4 * p), p), min=1e-7)
    z = torch.zeros_like(T)

    def population(a, lo, hi, share):
        n0, r = torch.exp(math.log(lo) + rnd[a] * math.log(hi / lo)), torch.exp(math.log(0.02) + rnd[a + 1] * math.log(50.0))
        sg = torch.log(1.1 + 0.5 * rnd[a + 2])
        m = [n0 * r ** k * torch.exp(0.5 * k * k * sg * sg) for k in range(4)]
        fits = torch.clamp(0.3 * Yv / (YL3 * m[3]), max=1.0)       # at most 30 % of the vapour's mass
        return [torch.where(rnd[a + 3] < share, x * fits, z) for x in m]

    ml, ms = population(3, 1e6, 1e13, 0.7), population(7, 1e5, 1e11, 0.5)
    soot = torch.where(rnd[11] < 0.8, 10.0 ** (9 + 4 * rnd[12]), z)
    return _cons(p, T, 450 * rnd[13], 20 * (rnd[14] - 0.5), Yv, ml, ms, soot / _gas(T, p, Yv)).T.contiguous()


def _rows(c, U):
    """Inputs, targets and masks of the surrogate in 64 bits for states U (n x 14)."""
    q, T, cv, _ = _prim(U.T)
    o = _rates(c, q, T, cv)
    ln, floor = lambda a: torch.log(torch.clamp(a, min=1e-30)), lambda a: torch.clamp(a, min=-30.0)  # noqa: E731
    lnsum = torch.logaddexp(o["lnJhom"], o["lnJhet"])
    l1p = torch.log1p(o["phi"])
    one, nuc = torch.ones_like(T), o["nuc"]
    Y = torch.stack([floor(lnsum - l1p), torch.log(torch.where(nuc, o["rc"], 1.0)), torch.asinh(o["Gl"]), torch.asinh(o["Gs"]), ln(o["xl"]),
                     ln(o["xs"]), floor(o["lnJhom"]), floor(o["lnJhet"]), l1p, o["Tl"] - T], -1)
    M = torch.stack([nuc * one, nuc * one, o["pl"] * one, o["ps"] * one, o["pl"] * one, o["ps"] * one, nuc * one, (nuc & o["soot"]) * one,
                     nuc * one, one], -1)
    return _features(c, q, T, o), torch.where(M > 0, Y, 0.0), M


def _surrogate_case(seed):
    return _params(dict(kind="mixing", nx=64, nr=32), seed)


def _train_rows(case, seed, dev):
    X, Y, M = _rows(_surrogate_case(seed), _visited(case["rows"], seed, dev))
    return [a.float().contiguous() for a in (X, Y, M)]


def _standard_rows(case, seed, dev):
    X, Y, M = _train_rows(case, seed, dev)
    one = lambda a: torch.where(a.std(0) > 1e-6, a.std(0), torch.ones_like(a[0]))  # noqa: E731
    return ((X - X.mean(0)) / one(X)).contiguous(), ((Y - Y.mean(0)) / one(Y) * M).contiguous(), M


def _train_cfg(case, seed):
    return dict(epochs=case["epochs"], batch=case["batch"], lr=2e-5, lr_final=1e-5, seed=seed, tensor_cores=int(case["tensor_cores"]),
                out_weight=[0.1, 0.1, 1.0, 1.0, 1.0, 1.0, 0.1, 0.1, 1.0, 0.1])


def _loss(p, X, Y, M, w):
    h, at = X, 0
    for l in range(5):
        i, n = LAYERS[l], LAYERS[l + 1]
        h = h @ p[at:at + i * n].view(n, i).T + p[at + i * n:at + i * n + n]
        h = h * torch.sigmoid(h) if l < 4 else h
        at += i * n + n
    return (w * (M * (h - Y)) ** 2).sum() / torch.clamp(M.sum(), min=1.0)


def _loss_grad(p, X, Y, M, w):
    p = p.detach().requires_grad_(True)
    with torch.enable_grad():
        loss = _loss(p, X, Y, M, w)
    return loss.detach(), torch.autograd.grad(loss, p)[0]


def _shuffle(n, state):
    """Fisher-Yates from splitmix64; returns the permutation and the generator's next state."""
    perm, mask = list(range(n)), (1 << 64) - 1
    for i in range(n - 1, 0, -1):
        state = (state + 0x9E3779B97F4A7C15) & mask
        z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        j = (z ^ (z >> 31)) % (i + 1)
        perm[i], perm[j] = perm[j], perm[i]
    return perm, state


def _finetune_exact(case, seed, dev):
    X, Y, M = (a.double() for a in _train_rows(case, seed, dev))
    cfg, p = _train_cfg(case, seed), torch.as_tensor(_weights()["params"].astype(np.float64), device=dev)
    w = torch.tensor(cfg["out_weight"], dtype=torch.float64, device=dev)

    def stats(A, K):
        n = torch.clamp(K.sum(0), min=1.0)
        mean = (A * K).sum(0) / n
        sd = torch.sqrt(torch.clamp((A * A * K).sum(0) / n - mean ** 2, min=0.0))
        sd = torch.where(sd > 1e-6, sd, 1.0)
        return torch.stack([mean, sd, torch.where(K > 0, A, INF).amin(0), torch.where(K > 0, A, -INF).amax(0)])

    sx, sy = stats(X, torch.ones_like(X)), stats(Y, M)
    X, Y = (X - sx[0]) / sx[1], (Y - sy[0]) / sy[1] * M
    b = min(cfg["batch"], X.shape[0])
    nb, m, v, t, rng, hist = X.shape[0] // b, torch.zeros_like(p), torch.zeros_like(p), 0, cfg["seed"], []
    for _ in range(cfg["epochs"]):
        perm, rng = _shuffle(X.shape[0], rng)
        perm, losses = torch.tensor(perm, device=dev), []
        for k in range(nb):
            i = perm[k * b:(k + 1) * b]
            loss, g = _loss_grad(p, X[i], Y[i], M[i], w)
            t += 1
            lr = cfg["lr_final"] + 0.5 * (cfg["lr"] - cfg["lr_final"]) * (1 + math.cos(math.pi * t / (cfg["epochs"] * nb)))
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - lr * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
            losses.append(loss)
        hist.append(torch.stack(losses).mean())
    return dict(params=p, inputs=sx.reshape(-1), targets=sy.reshape(-1), history=torch.stack(hist))


# ---- what the measuring program calls ---------------------------------------------------------------
def prepare(case, seed):
    dev, kind = "cuda", case["kind"]
    if kind in ("finetune", "gradient"):
        params = torch.tensor(_weights()["params"], device=dev)
        if kind == "finetune":
            X, Y, M = _train_rows(case, seed, dev)
            wb = P.ct_train_workspace_bytes(case["rows"], case["batch"], case["epochs"])
            return dict(case=case, X=X, Y=Y, M=M, start=params, params=params.clone(), cfg=_train_cfg(case, seed), wb=wb,
                        stats=torch.zeros(4 * 26, device=dev), work=torch.empty(wb // 4 + 64, device=dev))
        X, Y, M = _standard_rows(case, seed, dev)
        wb = P.ct_mlp_work_bytes(case["rows"])
        return dict(case=case, X=X, Y=Y, M=M, params=params, wb=wb, grad=torch.zeros_like(params),
                    loss=torch.zeros(1, device=dev), err=torch.zeros(1, dtype=torch.int32, device=dev), work=torch.empty(wb // 4 + 64, device=dev))
    if kind == "rates":
        return dict(case=case, flow=_surrogate_case(seed), U=_visited(case["rows"], seed, dev), blob=S.Surrogate.load(WEIGHTS).blob(dev),
                    out=torch.empty(case["rows"], 10, device=dev), err=torch.zeros(1, dtype=torch.int32, device=dev))
    prec = PRECISION[case["prec"]]
    dtype = torch.float64 if prec == FP64 else torch.float32
    blob = S.Surrogate.load(WEIGHTS).blob(dev) if prec == FP32_MLP else None
    if kind == "sweep":
        flows = _sweep(case, seed)
        rows = [_row_factors(c, seed + k) for k, c in enumerate(flows)]
        s = P.Batch(flows, rows, precision=prec, blob=blob)
        U0 = torch.cat([_state(c, r, seed + k, dev).to(dtype).reshape(-1) for k, (c, r) in enumerate(zip(flows, rows))])
    else:
        c = _params(case, seed)
        rows = _row_factors(c, seed)
        s = P.Solver(c, rows if c["geom"] == 1 else None, precision=prec)
        U0 = _state(c, rows, seed, dev).to(dtype)
        if blob is not None:
            s.attach_surrogate(blob)
    s.load_state(U0, CFL)
    if case.get("tune"):
        s.autotune()
    return dict(case=case, solver=s, U0=U0)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "finetune":
        state["params"].copy_(state["start"])
        hist = P.ct_train_surrogate(state["X"], state["Y"], state["M"], case["rows"], state["cfg"], state["params"], state["stats"],
                                    state["work"], state["wb"], torch.cuda.current_stream())
        return dict(params=state["params"], inputs=state["stats"][:64], targets=state["stats"][64:], history=hist.astype(np.float32))
    if kind == "gradient":
        a = (state["params"], state["X"], state["Y"], state["M"], case["rows"], state["grad"], state["loss"])
        stream = torch.cuda.current_stream()
        if case["tensor_cores"]:
            P.ct_mlp_loss_grad_tc(*a, state["err"], state["work"], state["wb"], stream)
        else:
            P.ct_mlp_loss_grad(*a, state["work"], state["wb"], stream)
        return dict(grad=state["grad"], loss=state["loss"])
    if kind == "rates":
        X, Y, M = S.dataset(state["flow"], state["U"])
        P.ct_mlp_infer(state["blob"], X, case["rows"], state["out"], state["err"], torch.cuda.current_stream())
        return dict(inputs=X, targets=Y, masks=M, predicted=state["out"])
    s = state["solver"]
    s.load_state(state["U0"], CFL)
    s.step(case["steps"], CFL)
    if kind == "sweep":
        return [_fields(s.state(k)) for k in range(case["cases"])]
    return _fields(s.U)


def work(case):
    """Bytes of one pass: its inputs once and its outputs once. Operations: those of the method (the flow's finite-volume
    stage with exact zeros skipped, two stages a step; a network evaluation; forward, input and weight gradients)."""
    kind = case["kind"]
    if kind in ("finetune", "gradient"):
        n = case["rows"] * case.get("epochs", 1)
        return dict(bytes=case["rows"] * 36 * 4.0 + 2 * 4 * 53000.0, flops=6.0 * MACS * n)
    if kind == "rates":
        return dict(bytes=case["rows"] * (14 * 8.0 + 46 * 4.0), flops=case["rows"] * (2.0 * MACS + 1500.0))
    cells = sum(c["nx"] * c["nr"] for c in _sweep(case, 0)) if kind == "sweep" else case["nx"] * case["nr"]
    nf = 18 if case.get("bimodal") else 14
    per = 1250.0 if case.get("viscous") else 565.0
    return dict(bytes=2.0 * cells * nf * (8 if case["prec"] == "fp64" else 4), flops=2 * per * cells * case["steps"])


def exact(case, seed):
    dev, kind = _dev(), case["kind"]
    with torch.no_grad():
        if kind == "finetune":
            return _finetune_exact(case, seed, dev)
        if kind == "gradient":
            X, Y, M = (a.double() for a in _standard_rows(case, seed, dev))
            p = torch.as_tensor(_weights()["params"].astype(np.float64), device=dev)
            loss, g = _loss_grad(p, X, Y, M, torch.ones(10, dtype=torch.float64, device=dev))
            return dict(grad=g, loss=loss.reshape(1))
        if kind == "rates":
            X, Y, M = _rows(_surrogate_case(seed), _visited(case["rows"], seed, dev))
            return dict(inputs=X, targets=Y, masks=M, predicted=_network(_weights(), X, dev))
        dtype = torch.float64 if case["prec"] == "fp64" else torch.float32
        z = _weights() if case["prec"] == "surrogate" else None
        if kind == "sweep":
            flows, out = _sweep(case, seed), []
            for k, c in enumerate(flows):
                rows = _row_factors(c, seed + k)
                out.append(_fields(_advance(c, rows, _state(c, rows, seed + k, dev).to(dtype), case["steps"], z)))
            return out
        c = _params(case, seed)
        rows = _row_factors(c, seed)
        return _fields(_advance(c, rows, _state(c, rows, seed, dev).to(dtype), case["steps"], z))
