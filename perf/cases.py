"""Performance cases of the property engine: what a flow solver and a surrogate
training run ask of it, through the Python entry points.

A solver calls, per time step and mesh block, the temperature from enthalpy,
the properties at that temperature, the per-species quantities, or a surrogate
in their place; the sizes run from a boundary patch of a thousand cells to the
256^3 field of ``bench.py``.  Training runs steps of one batch size on a
labelled pool.  Cell states are of two kinds, as in
``paper_2312_04830_gb300/workloads.py``: "field", the flame-vortex field in
grid order (neighbouring cells alike), and "scattered", independent cells over
the whole state space (as gathered from a mesh).  ``exact`` evaluates the same
methods in plain FP64 torch.
"""
import math

import numpy as np
import torch

from paper_2312_04830_gb300 import binding, workloads

SPECIES_TABLE = workloads.species_table()
NS = SPECIES_TABLE.n
R = 8.314462618
P_REF = workloads.P_REF
OUT6 = ("rho", "Z", "h", "cp", "mu", "lambda")
OUT8 = OUT6 + ("psi", "alpha")
OUT_INVERSE = ("T", "rho", "psi", "mu", "alpha", "cp")


def listed():
    return [
        # a boundary patch or a small mesh block: the call's latency
        {"name": "props_fp64_patch", "op": "props", "precision": "fp64", "n": 1000, "cells": "scattered"},
        # FP64 properties of a 128^3 mesh block (the solver's accurate path)
        {"name": "props_fp64_block", "op": "props", "precision": "fp64", "n": 128 ** 3, "cells": "field"},
        # FP32 properties of the whole 256^3 field
        {"name": "props_fp32_field", "op": "props", "precision": "fp32", "n": 256 ** 3, "cells": "field"},
        # mixed precision with the compressibility psi and lambda/cp, an odd gathered cell list
        {"name": "props_ext_mixed_odd", "op": "props_ext", "precision": "mixed", "n": 1000003, "cells": "scattered"},
        # the inversion T(h, p, Y) after an enthalpy step, in the three precisions
        {"name": "T_from_h_fp64_block", "op": "T_from_h", "precision": "fp64", "n": 128 ** 3, "cells": "field"},
        {"name": "T_from_h_fp32_odd", "op": "T_from_h", "precision": "fp32", "n": 4500001, "cells": "field"},
        {"name": "T_from_h_mixed_odd", "op": "T_from_h", "precision": "mixed", "n": 300007, "cells": "scattered"},
        # per-species enthalpies and diffusion coefficients for the species equations
        {"name": "species_fp64_block", "op": "species", "precision": "fp64", "n": 64 ** 3, "cells": "field"},
        {"name": "species_fp32_odd", "op": "species", "precision": "fp32", "n": 2000003, "cells": "scattered"},
        # the surrogate in the property call's place, with its low-confidence tests
        {"name": "infer_forward_large", "op": "infer", "mode": "forward", "width": 512, "layers": 4, "n": 1 << 22,
         "cells": "field", "chunk": 1 << 22, "confidence": 0.2},
        # the paper's arrangement (h, p, Y in), three hidden layers, one small block
        {"name": "infer_inverse_small", "op": "infer", "mode": "inverse", "width": 256, "layers": 3, "n": 20011,
         "cells": "field", "chunk": 1 << 20, "confidence": 0.0},
        # training at the training configuration's batch, and the weights handed over after a few steps
        {"name": "train_512x4", "op": "train", "mode": "forward", "width": 512, "layers": 4, "batch": 65536,
         "steps": 8, "pool": 1 << 20},
    ]


def draw(rng):
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n + rng.randrange(0, 3)

    op = rng.choice(["props", "props", "props_ext", "T_from_h", "T_from_h", "species", "infer", "infer", "train"])
    if op in ("props", "props_ext", "T_from_h", "species"):
        precision = rng.choice(["fp64", "fp64", "fp32", "mixed"])
        top = {"props": 1 << 21, "props_ext": 1 << 21, "T_from_h": 1 << 21, "species": 1 << 18}[op]
        if precision != "fp64":
            top *= 2
        return {"op": op, "precision": precision, "n": size(1000, top), "cells": rng.choice(["field", "scattered"])}
    if op == "infer":
        mode = rng.choice(["forward", "inverse"])
        return {"op": op, "mode": mode, "width": rng.choice([256, 512]), "layers": rng.choice([3, 4]),
                "n": size(1000, 1 << 21), "cells": "field", "chunk": rng.choice([1 << 18, 1 << 20, 1 << 22]),
                "confidence": rng.choice([0.0, 0.2 if mode == "forward" else 0.5])}
    return {"op": op, "mode": rng.choice(["forward", "inverse"]), "width": rng.choice([256, 512]),
            "layers": rng.choice([3, 4]), "batch": 128 * size(8, 448), "steps": rng.choice([1, 4, 8]), "pool": 1 << 20}


# ------------------------------------------------------------- cell states
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _dirichlet_half(n, g):
    z = torch.randn((NS, n), generator=g, device="cuda", dtype=torch.float64)
    z *= z
    return z / z.sum(dim=0, keepdim=True)


def _flame_sheet(Z):
    """T and Y of a Burke-Schumann CH4/O2 flame sheet at mixture fraction Z."""
    z_st, f_co2 = workloads._stoich()
    lean = Z <= z_st
    Y = torch.zeros((NS, Z.numel()), dtype=torch.float64, device=Z.device)
    yp = torch.where(lean, Z / z_st, (1.0 - Z) / (1.0 - z_st))
    zero = torch.zeros_like(Z)
    Y[1] = torch.where(lean, 1.0 - Z / z_st, zero)
    Y[0] = torch.where(lean, zero, (Z - z_st) / (1.0 - z_st))
    Y[2] = f_co2 * yp
    Y[3] = (1.0 - f_co2) * yp
    T = torch.where(lean, workloads.T_OX + (workloads.T_ST - workloads.T_OX) * Z / z_st,
                    workloads.T_FUEL + (workloads.T_ST - workloads.T_FUEL) * (1.0 - Z) / (1.0 - z_st))
    return T, Y


def _scattered_cells(n, g):
    T = 100.0 + 3400.0 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    p = P_REF * (0.95 + 0.1 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64))
    return T, p, _dirichlet_half(n, g)


def _field_cells(n, g):
    """The first n cells of a flame-vortex field, z fastest; the vortex's phase,
    the flame's place and the pressure wave come from the generator."""
    edge = max(2, int(math.ceil(n ** (1.0 / 3.0) - 1e-9)))
    ph = torch.rand(4, generator=g, device="cuda", dtype=torch.float64)
    i = torch.arange(n, device="cuda")
    layers = -(-n // (edge * edge))
    x = (torch.div(i, edge * edge, rounding_mode="floor").double() + 0.5) / layers
    y = (torch.div(i, edge, rounding_mode="floor") % edge + 0.5).double() / edge
    z = (i % edge + 0.5).double() / edge
    del i
    wave = torch.cos(2 * math.pi * (y + ph[0])) * torch.cos(2 * math.pi * (z + ph[1]))
    xp = (x - 0.5 + 0.05 * (ph[2] - 0.5)) + 0.3 * wave
    T, Y = _flame_sheet(0.5 * (1.0 + torch.tanh(40.0 * xp)))
    p = P_REF * (1.0 + 0.02 * torch.cos(2 * math.pi * (x + ph[3])) * wave)
    return T, p, Y


def _physical(T, p, Y):
    """The states whose outcome is physical, as the training pool's rule has it (``train.label_pool``):
    a cell whose viscosity or conductivity falls below the dilute gas's, or which lies next to a pole
    of Chung's dense terms (where a change of 1e-4 in its state moves them by over 0.3 %), takes the
    state of the last cell before it that does not."""
    dense, dilute = _properties(T, p, Y), _properties(T, torch.ones_like(p), Y)
    Yn = Y * (1.0 + 1e-4 * torch.tensor([(-1.0) ** k for k in range(NS)], device=Y.device, dtype=Y.dtype)[:, None])
    near = _properties(T * (1.0 + 1e-4), p, Yn / Yn.sum(dim=0, keepdim=True))
    good = torch.ones_like(T, dtype=torch.bool)
    for k in ("mu", "lambda"):
        good &= (dense[k] >= 0.9 * dilute[k]) & ((near[k] / dense[k] - 1.0).abs() <= 3e-3)
    i = torch.where(good, torch.arange(T.numel(), device=T.device), -1)
    i = torch.cummax(i, dim=0).values
    i = torch.where(i < 0, good.to(torch.uint8).argmax(), i)
    return T[i], p[i], Y[:, i].contiguous()


def _cells(case, seed):
    g = _generator(seed)
    T, p, Y = _physical(*(_field_cells if case["cells"] == "field" else _scattered_cells)(case["n"], g))
    return T, p, Y, g


def _training_states(n, g):
    """Half scattered cells, half flame-sheet states with noise (half of them in composition too)."""
    Tu, pu, Yu = _scattered_cells(n // 2, g)
    m = n - n // 2
    Z = torch.rand(m, generator=g, device="cuda", dtype=torch.float64)
    thin = 0.5 * (1.0 + torch.tanh(10.0 * torch.rand(m, generator=g, device="cuda", dtype=torch.float64) - 5.0))
    Z = torch.where(torch.rand(m, generator=g, device="cuda") < 0.5, thin, Z)
    T, Y = _flame_sheet(Z)
    T = (T * (1.0 + 0.03 * torch.randn(m, generator=g, device="cuda", dtype=torch.float64))).clamp(100.0, 3500.0)
    Y = Y + 0.02 * _dirichlet_half(m, g) * (torch.rand(m, generator=g, device="cuda") < 0.5)
    Y /= Y.sum(dim=0, keepdim=True)
    p = P_REF * (0.95 + 0.1 * torch.rand(m, generator=g, device="cuda", dtype=torch.float64))
    return _physical(torch.cat([Tu, T]), torch.cat([pu, p]), torch.cat([Yu, Y], dim=1))


# ------------------------------------------- the methods in plain FP64 torch
def _omegas():
    b = 0.07779607390388846
    zc = (1.0 - b) / 3.0
    return 3.0 * zc * zc + 3.0 * b * b + 2.0 * b, b


def _cubic_roots(c2, c1, c0):
    """The three roots of Z^3 + c2 Z^2 + c1 Z + c0 (-inf where there is no real one)."""
    P = c1 - c2 * c2 / 3.0
    Q = 2.0 * (c2 / 3.0) ** 3 - c2 * c1 / 3.0 + c0
    disc = 0.25 * Q * Q + (P / 3.0) ** 3
    sq = torch.sqrt(disc.clamp_min(0.0))
    t = -0.5 * Q - torch.copysign(sq, 0.5 * Q)
    u = torch.copysign(t.abs() ** (1.0 / 3.0), t)
    one = u - P / (3.0 * torch.where(u == 0, torch.ones_like(u), u)) - c2 / 3.0
    m = 2.0 * torch.sqrt((-P / 3.0).clamp_min(0.0))
    arg = (3.0 * Q / torch.where(P * m == 0, torch.ones_like(P), P * m)).clamp(-1.0, 1.0)
    th = torch.acos(arg) / 3.0
    none = torch.full_like(P, -math.inf)
    roots = [torch.where(disc > 0, one, m * torch.cos(th) - c2 / 3.0)]
    roots += [torch.where(disc > 0, none, m * torch.cos(th + s) - c2 / 3.0)
              for s in (4.0 * math.pi / 3.0, 2.0 * math.pi / 3.0)]
    for k in range(3):
        z = roots[k]
        for _ in range(4):
            d = (3.0 * z + 2.0 * c2) * z + c1
            dz = (((z + c2) * z + c1) * z + c0) / torch.where(d == 0, torch.ones_like(d), d)
            z = torch.where(torch.isfinite(z), z - dz, z)
        roots[k] = z
    return roots


def _col(a, like):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device=like.device)


def _thermo(T, p, Y, want_cp=True):
    """Peng-Robinson with van der Waals mixing and NASA-7 ideal-gas terms (Sec. 2)."""
    sp = SPECIES_TABLE
    moles = sum(Y[k] / (sp.W[k] * 1e-3) for k in range(NS))
    X = [Y[k] / (sp.W[k] * 1e-3) / moles for k in range(NS)]
    W = 1.0 / moles
    oa, ob = _omegas()
    s0, s1, s2, bm = (torch.zeros_like(T) for _ in range(4))
    sqT = torch.sqrt(T)
    for k in range(NS):
        w = sp.omega[k]
        ac, kap = math.sqrt(oa) * R * sp.Tc[k] / math.sqrt(sp.pc[k]), 0.37464 + 1.54226 * w - 0.26992 * w * w
        u = 1.0 + kap * (1.0 - sqT / math.sqrt(sp.Tc[k]))
        xg = torch.where(u >= 0, ac * X[k], -ac * X[k])
        s0 += xg * u
        s1 += xg * (-0.5 * kap / math.sqrt(sp.Tc[k])) / sqT
        s2 += xg * (0.25 * kap / math.sqrt(sp.Tc[k])) / (sqT * T)
        bm += X[k] * (ob * R * sp.Tc[k] / sp.pc[k])
    am, dam, d2am = s0 * s0, 2.0 * s0 * s1, 2.0 * (s0 * s2 + s1 * s1)
    RT = R * T
    A, B = am * p / (RT * RT), bm * p / RT
    roots = _cubic_roots(B - 1.0, A - 3.0 * B * B - 2.0 * B, B * B + B ** 3 - A * B)
    r2 = math.sqrt(2.0)
    Z, best = roots[0], None
    for z in roots:
        ok = z > B
        zs = torch.where(ok, z, B + 1.0)
        gr = zs - 1.0 - torch.log(zs - B) - A / (2 * r2 * B) * torch.log((zs + (1 + r2) * B) / (zs + (1 - r2) * B))
        gr = torch.where(ok, gr, torch.full_like(gr, math.inf))
        if best is None:
            best = gr
        else:
            take = gr < best
            Z, best = torch.where(take, z, Z), torch.where(take, gr, best)
    cp_ig, h_ig = torch.zeros_like(T), torch.zeros_like(T)
    for k in range(NS):
        lo = T < sp.T_mid[k]
        a = [torch.where(lo, torch.full_like(T, sp.nasa_lo[k, j]), torch.full_like(T, sp.nasa_hi[k, j])) for j in range(6)]
        cp_ig += X[k] * R * ((((a[4] * T + a[3]) * T + a[2]) * T + a[1]) * T + a[0])
        h_ig += X[k] * R * (((((a[4] / 5 * T + a[3] / 4) * T + a[2] / 3) * T + a[1] / 2) * T + a[0]) * T + a[5])
    V = Z * RT / p
    L = torch.log1p(2 * r2 * B / (Z + (1 - r2) * B))
    h = (h_ig + RT * (Z - 1.0) + (T * dam - am) / (2 * r2 * bm) * L) / W
    den = V * V + 2.0 * bm * V - bm * bm
    dpdT = R / (V - bm) - dam / den
    dpdV = -RT / (V - bm) ** 2 + 2.0 * am * (V + bm) / den ** 2
    cp = (cp_ig + T * d2am / (2 * r2 * bm) * L - T * dpdT * dpdT / dpdV - R) / W
    return {"X": X, "W": W, "Z": Z, "h": h, "cp": cp, "rho": p * W / (Z * RT), "rho_mol": 1.0 / V, "cv": cp_ig - R,
            "dpdT": dpdT, "dpdV": dpdV}


CHUNG_E = ((6.324, 50.412, -51.680, 1189.0), (1.210e-3, -1.154e-3, -6.257e-3, 0.03728),
           (5.283, 254.209, -168.48, 3898.0), (6.623, 38.096, -8.464, 31.42), (19.745, 7.630, -14.354, 31.53),
           (-1.900, -12.537, 4.985, -18.15), (24.275, 3.450, -11.291, 69.35), (0.7972, 1.117, 0.01235, -4.117),
           (-0.2382, 0.06770, -0.8163, 4.025), (0.06863, 0.3479, 0.5926, -0.727))
CHUNG_B = ((2.4166, 0.74824, -0.91858, 121.72), (-0.50924, -1.5094, -49.991, 69.983),
           (6.6107, 5.6207, 64.760, 27.039), (14.543, -8.9139, -5.6379, 74.344), (0.79274, 0.82019, -0.69369, 6.3173),
           (-5.8634, 12.801, 9.5893, 65.529), (91.089, 128.11, -54.217, 523.81))


def _chung(T, t):
    """Chung's dense-fluid viscosity and conductivity with his mixture rules (Sec. 2)."""
    sp, X = SPECIES_TABLE, t["X"]
    sig, eps = 0.809 * np.cbrt(sp.Vc), sp.Tc / 1.2593
    s3, e3, m2, w3, mu, kp = (torch.zeros_like(T) for _ in range(6))
    for i in range(NS):
        for j in range(i, NS):
            xx = X[i] * X[j] * (1.0 if i == j else 2.0)
            s, e = math.sqrt(sig[i] * sig[j]), math.sqrt(eps[i] * eps[j])
            s3 += xx * s ** 3
            e3 += xx * (e * s ** 3)
            m2 += xx * (e * s * s * math.sqrt(2.0 * sp.W[i] * sp.W[j] / (sp.W[i] + sp.W[j])))
            w3 += xx * (0.5 * (sp.omega[i] + sp.omega[j]) * s ** 3)
            if sp.dipole[i] * sp.dipole[j] != 0:
                mu += xx * ((sp.dipole[i] * sp.dipole[j]) ** 2 / s ** 3)
            if sp.kappa[i] * sp.kappa[j] != 0:
                kp += xx * math.sqrt(sp.kappa[i] * sp.kappa[j])
    em, w, mu4 = e3 / s3, w3 / s3, s3 * mu
    M = (m2 / (em * s3 ** (2.0 / 3.0))) ** 2
    Vc, Tc = s3 / 0.809 ** 3, 1.2593 * em
    mur4 = mu4 * (131.3 ** 2 / (Vc * Tc)) ** 2
    Ts, Tr = 1.2593 * T / Tc, T / Tc
    Fc = 1.0 - 0.2756 * w + 0.059035 * mur4 + kp
    Ov = 1.16145 * Ts ** -0.14874 + 0.52487 * torch.exp(-0.77320 * Ts) + 2.16178 * torch.exp(-2.43787 * Ts)
    y = t["rho_mol"] * 1e-6 * Vc / 6.0
    G1 = (1.0 - 0.5 * y) / (1.0 - y) ** 3
    E = [c[0] + c[1] * w + c[2] * mur4 + c[3] * kp for c in CHUNG_E]
    B = [c[0] + c[1] * w + c[2] * mur4 + c[3] * kp for c in CHUNG_B]
    G2 = (E[0] * (-torch.expm1(-E[3] * y) / y) + E[1] * G1 * torch.exp(E[4] * y) + E[2] * G1) / (E[0] * E[3] + E[1] + E[2])
    ess = E[6] * y * y * G2 * torch.exp(E[7] + E[8] / Ts + E[9] / (Ts * Ts))
    V23 = Vc ** (2.0 / 3.0)
    visc = (torch.sqrt(Ts) / Ov * Fc * (1.0 / G2 + E[5] * y) + ess) * 36.344e-7 * torch.sqrt(M * Tc) / V23
    eta0 = 40.785e-7 * Fc * torch.sqrt(M * T) / (V23 * Ov)
    H2 = (B[0] * (-torch.expm1(-B[3] * y) / y) + B[1] * G1 * torch.exp(B[4] * y) + B[2] * G1) / (B[0] * B[3] + B[1] + B[2])
    al, be, Zp = t["cv"] / R - 1.5, 0.7862 - 0.7109 * w + 1.3168 * w * w, 2.0 + 10.5 * Tr * Tr
    Psi = 1.0 + al * ((0.215 + 0.28288 * al - 1.061 * be + 0.26665 * Zp) / (0.6366 + be * Zp + 1.061 * al * be))
    q = 3.586e-3 * torch.sqrt(Tc / (M * 1e-3)) / V23
    lam = 31.2 * eta0 * Psi / (M * 1e-3) * (1.0 / H2 + B[5] * y) + q * B[6] * y * y * torch.sqrt(Tr) * H2
    return visc, lam


def _properties(T, p, Y):
    """All eight outputs of the forward call, and T."""
    t = _thermo(T, p, Y)
    mu, lam = _chung(T, t)
    V = 1.0 / t["rho_mol"]
    dVdT = -t["dpdT"] / t["dpdV"]
    drho_p, drho_T = -t["W"] / V ** 2 / t["dpdV"], -t["W"] / V ** 2 * dVdT
    psi = drho_p - drho_T * (V - T * dVdT) / (t["cp"] * t["W"])
    return {"rho": t["rho"], "Z": t["Z"], "h": t["h"], "cp": t["cp"], "mu": mu, "lambda": lam, "psi": psi,
            "alpha": lam / t["cp"], "T": T}


def _temperature(h, p, Y, T):
    """T(h, p, Y) by Newton from a temperature next to the root."""
    for _ in range(8):
        t = _thermo(T, p, Y)
        T = T - (t["h"] - h) / t["cp"]
    return T


def _species(T, p, Y):
    """h_k / (R T) and mixture-averaged D_k (Chapman-Enskog with Neufeld's collision integral)."""
    sp = SPECIES_TABLE
    moles = sum(Y[k] / (sp.W[k] * 1e-3) for k in range(NS))
    X = [Y[k] / (sp.W[k] * 1e-3) / moles for k in range(NS)]
    hk, acc = [], [torch.zeros_like(T) for _ in range(NS)]
    own = []
    for k in range(NS):
        lo = T < sp.T_mid[k]
        a = [torch.where(lo, torch.full_like(T, sp.nasa_lo[k, j]), torch.full_like(T, sp.nasa_hi[k, j])) for j in range(6)]
        hk.append((((a[4] / 5 * T + a[3] / 4) * T + a[2] / 3) * T + a[1] / 2) * T + a[0] + a[5] / T)
        for j in range(k, NS):
            s = 0.5 * 0.809 * (sp.Vc[k] ** (1.0 / 3.0) + sp.Vc[j] ** (1.0 / 3.0))
            Ts = T / math.sqrt(sp.Tc[k] * sp.Tc[j] / 1.2593 ** 2)
            om = 1.06036 * Ts ** -0.15610 + 0.19300 * torch.exp(-0.47635 * Ts) + 1.03587 * torch.exp(-1.52996 * Ts) \
                + 1.76474 * torch.exp(-3.89411 * Ts)
            inv = om * p * (s * s * math.sqrt(2.0 / (1.0 / sp.W[k] + 1.0 / sp.W[j])) / 0.0266) / T ** 1.5
            if j == k:
                own.append(1.0 / inv)
            else:
                acc[k] += X[j] * inv
                acc[j] += X[k] * inv
    total = sum(Y[k] for k in range(NS))
    D = []
    for k in range(NS):
        others = sum(Y[j] for j in range(NS) if j != k) / total
        D.append(torch.where(acc[k] > 0, others / torch.where(acc[k] > 0, acc[k], torch.ones_like(T)), own[k]))
    return torch.stack(hk), torch.stack(D)


# ----------------------------------------------------------------- networks
def _h_ideal(T, Y):
    sp = SPECIES_TABLE
    h = torch.zeros_like(Y[0])
    for k in range(NS):
        lo = T < sp.T_mid[k]
        a = [torch.where(lo, torch.full_like(T, sp.nasa_lo[k, j]), torch.full_like(T, sp.nasa_hi[k, j])) for j in range(6)]
        h += Y[k] / (sp.W[k] * 1e-3) * R * \
            (((((a[4] / 5 * T + a[3] / 4) * T + a[2] / 3) * T + a[1] / 2) * T + a[0]) * T + a[5])
    return h


def _features(mode, v, p, Y):
    """The network's 13 inputs from T (forward) or h (inverse), p and Y."""
    sp = SPECIES_TABLE
    n = [Y[k] / (sp.W[k] * 1e-3) for k in range(NS)]
    s = sum(n)
    Tpc = sum(n[k] * sp.Tc[k] for k in range(NS)) / s
    if mode == "forward":
        first, derived = torch.log(v), Tpc / v
    else:
        first, derived = v - _h_ideal(torch.full_like(v, 298.15), Y), torch.log(Tpc)
    return torch.stack([first, p] + [Y[k] for k in range(NS)] + [derived, -torch.log(s)])


def _targets(mode, v, Y, y):
    if mode == "forward":
        return torch.stack([torch.log(y[0]), y[1], y[2] - _h_ideal(v, Y), torch.log(y[3]), torch.log(y[4]), torch.log(y[5])])
    return torch.log(y)


def _gelu(z):
    return 0.5 * z * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (z + 0.044715 * z ** 3)))


def _forward(layers, x):
    for W, b in layers[:-1]:
        x = _gelu(x @ W.T + b)
    return x @ layers[-1][0].T + layers[-1][1]


def _pool(mode, n, g):
    """Labelled states as a training run holds them: x [11, n] and y [6, n] in FP32."""
    T, p, Y = _training_states(n, g)
    o = _properties(T, p, Y)
    if mode == "forward":
        return torch.cat([T[None], p[None], Y]).float(), torch.stack([o[k] for k in OUT6]).float()
    return torch.cat([o["h"][None], p[None], Y]).float(), torch.stack([o[k] for k in OUT_INVERSE]).float()


def _model(case, x, y, g, fitted):
    """Weights and normalisation of a model: hidden layers drawn by He's rule; with
    `fitted`, an output layer fitted to the pool by least squares (so that the
    outputs are those of a usable model), else a drawn one (training's start)."""
    mode, W, L = case["mode"], case["width"], case["layers"]
    xd, yd = x.double(), y.double()
    f, q = _features(mode, xd[0], xd[1], xd[2:]), _targets(mode, xd[0], xd[2:], yd)
    lo, hi = f.min(dim=1).values, f.max(dim=1).values
    w = 0.01 * (hi - lo)
    norm = np.zeros(binding.SG_NORM_FLOATS, dtype=np.float32)
    fm, fs, qm, qs = f.mean(dim=1), f.std(dim=1), q.mean(dim=1), q.std(dim=1)
    norm[:64] = torch.cat([fm, fs, qm, qs, lo - w, hi + w]).float().cpu().numpy()
    norm[74:] = 1.0
    layers, a = [], ((f - fm[:, None]) / fs[:, None])[:, ::4][:, :16384].T
    t = ((q - qm[:, None]) / qs[:, None])[:, ::4][:, :16384].T
    for l in range(L):
        n_in = a.shape[1]
        Wl = torch.randn((W, n_in), generator=g, device="cuda") * math.sqrt((1.0 if l == 0 else 2.0) / n_in)
        bl = 0.3 * torch.randn(W, generator=g, device="cuda")
        layers.append((Wl, bl))
        a = _gelu(a @ Wl.double().T + bl.double())
    if fitted:
        F = torch.cat([a, torch.ones_like(a[:, :1])], dim=1)
        weight = torch.ones_like(F[:, :1])
        weight[F.shape[0] // 2:] = 30.0   # the pool's flame-sheet half
        S = F.T @ (weight * F)
        S.diagonal().add_(1e-5 * S.diagonal().mean())
        c = torch.linalg.solve(S, F.T @ (weight * t))
        layers.append((c[:W].T.float().contiguous(), c[W].float()))
    else:
        layers.append((torch.randn((6, W), generator=g, device="cuda") / math.sqrt(W), torch.zeros(6, device="cuda")))
    flat = torch.cat([v.reshape(-1) for wb in layers for v in wb]).cpu().numpy()
    return layers, norm, flat


def _surrogate(case, ctx, norm, flat):
    sg = binding.Surrogate(ctx, width=case["width"], hidden_layers=case["layers"], max_batch=case.get("batch", 128),
                           infer_chunk=case.get("chunk", 128))
    sg.set_mode(case["mode"])
    sg.set_normalization(norm)
    sg.set_params(flat)
    c = case.get("confidence", 0.0)
    if c and case["mode"] == "forward":
        sg.set_confidence(c)
    if c:
        sg.set_transport_confidence(c)
    return sg


def _network(case, seed):
    """A fitted model's layers, normalisation and flat parameters (another seed, another model)."""
    g = _generator(1000 + seed)
    x, y = _pool(case["mode"], 1 << 16, g)
    return _model(case, x, y, g, True)


# --------------------------------------------------------------- the passes
def prepare(case, seed):
    op = case["op"]
    s = {"op": op, "case": case, "ctx": binding.PropertyContext(SPECIES_TABLE)}
    if op == "train":
        g = _generator(seed)
        x, y = _pool(case["mode"], case["pool"], g)
        layers, norm, flat = _model(case, x, y, g, False)
        s.update(x=x, y=y, sg=_surrogate(case, s["ctx"], norm, flat), loss=torch.empty(case["steps"], device="cuda"))
        return s
    T, p, Y, g = _cells(case, seed)
    if op == "infer":
        v = T if case["mode"] == "forward" else _thermo(T, p, Y)["h"]
        _, norm, flat = _network(case, seed)
        s.update(v=v.float(), p=p.float(), Y=Y.float(), sg=_surrogate(case, s["ctx"], norm, flat))
        return s
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    s.update(precision=case["precision"], p=p.to(dt), Y=Y.to(dt))
    if op == "T_from_h":
        s.update(h=_thermo(_true_T(T, g), p, Y)["h"].to(dt), guess=T.to(dt))
    else:
        s["T"] = T.to(dt)
    return s


def _true_T(T, g):
    return (T * (0.95 + 0.1 * torch.rand(T.numel(), generator=g, device="cuda", dtype=torch.float64))).clamp(100.0, 3500.0)


def run(state):
    op, ctx = state["op"], state["ctx"]
    if op == "props":
        out, status = ctx.props(state["T"], state["p"], state["Y"], state["precision"])
        return {**{k: out[i] for i, k in enumerate(OUT6)}, "status": status}
    if op == "props_ext":
        out, status = ctx.props_ext(state["T"], state["p"], state["Y"], state["precision"])
        return {**{k: out[i] for i, k in enumerate(OUT8)}, "status": status}
    if op == "T_from_h":
        # the third result counts the work done per cell, not a property of it
        T, status, _ = ctx.T_from_h(state["h"], state["p"], state["Y"], state["guess"], state["precision"])
        return {"T": T, "status": status}
    if op == "species":
        hk, Dk, status = ctx.species_props(state["T"], state["p"], state["Y"], state["precision"])
        return {"hk": hk, "Dk": Dk, "status": status}
    if op == "infer":
        out, fallback = state["sg"].infer(state["v"], state["p"], state["Y"])
        names = OUT6 if state["case"]["mode"] == "forward" else OUT_INVERSE
        return {**{k: out[i] for i, k in enumerate(names)}, "fallback": fallback}
    c, sg, loss = state["case"], state["sg"], state["loss"]
    for k in range(c["steps"]):
        sg.train_step(state["x"], state["y"], c["batch"], 1e-3, sample_seed=k + 1, loss_out=loss[k:])
    return {"loss": loss, "params": sg.get_params()}


def work(case):
    op = case["op"]
    if op in ("infer", "train"):
        W, L = case["width"], case["layers"]
        mlp = 2.0 * (13 * W + (L - 1) * W * W + 6 * W)
        if op == "infer":
            return {"bytes": case["n"] * (11 * 4 + 6 * 4 + 1), "flops": case["n"] * mlp}
        rows = case["batch"] * case["steps"]
        params = 13 * W + (L - 1) * W * W + 6 * W + L * W + 6
        return {"bytes": rows * 17 * 4 + case["steps"] * params * 24, "flops": 3.0 * rows * mlp}
    es, n = (8 if case["precision"] == "fp64" else 4), case["n"]
    outs = {"props": 6, "props_ext": 8, "T_from_h": 1, "species": 18}[op]
    ins = 12 if op == "T_from_h" else 11
    # floating-point operations of one evaluation per cell (divisions, roots and
    # exponentials weighted by what they cost), one for the inversion
    flops = {"props": 1700, "props_ext": 1730, "T_from_h": 520, "species": 4100}[op]
    return {"bytes": n * ((ins + outs) * es + 4), "flops": float(n * flops)}


# ------------------------------------------------------- the answers in FP64
def exact(case, seed):
    op = case["op"]
    if op == "train":
        return _exact_train(case, seed)
    T, p, Y, g = _cells(case, seed)
    if op == "infer":
        return _exact_infer(case, seed, T, p, Y)
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    # the inputs as the call gets them
    Tc, pc, Yc = T.to(dt).double(), p.to(dt).double(), Y.to(dt).double()
    if op == "T_from_h":
        Tt = _true_T(T, g)
        h = _thermo(Tt, p, Y)["h"].to(dt).double()
        return {"T": Tt if dt == torch.float64 else _temperature(h, pc, Yc, Tt), "status": None}
    if op == "species":
        hk, Dk = _species(Tc, pc, Yc)
        return {"hk": hk, "Dk": Dk, "status": None}
    o = _properties(Tc, pc, Yc)
    return {**{k: o[k] for k in (OUT6 if op == "props" else OUT8)}, "status": None}


def _exact_infer(case, seed, T, p, Y):
    mode = case["mode"]
    v = (T if mode == "forward" else _thermo(T, p, Y)["h"]).float().double()
    p, Y = p.float().double(), Y.float().double()
    layers, norm, _ = _network(case, seed)
    layers = [(W.double(), b.double()) for W, b in layers]
    nm = _col(norm, v)
    f = _features(mode, v, p, Y)
    lo, hi = nm[38:51, None], nm[51:64, None]
    out = ((f < lo) | (f > hi)).any(dim=0)
    x = ((f - nm[:13, None]) / nm[13:26, None]).T
    q = torch.cat([_forward(layers, x[a:a + (1 << 19)]) for a in range(0, x.shape[0], 1 << 19)])
    q = (q * nm[32:38] + nm[26:32]).T
    if mode == "forward":
        net = torch.stack([q[0].exp(), q[1], q[2] + _h_ideal(v, Y), q[3].exp(), q[4].exp(), q[5].exp()])
        Tn, rho, mu, lam = v, net[0], net[4], net[5]
    else:
        net = q.exp()
        Tn, rho, mu, lam = net[0], net[1], net[3], net[4] * net[5]
    c = case["confidence"]
    t = _thermo(Tn.clamp(60.0, 5000.0), p, Y)
    if c and mode == "forward":
        out |= ~((rho * net[1] * R * v / (p * t["W"]) - 1.0).abs() <= c)
    if c:
        t["rho_mol"] = rho / t["W"]
        mc, lc = _chung(Tn, t)
        out |= ~((mu - mc).abs() <= c * mc.abs()) | ~((lam - lc).abs() <= c * lc.abs())
    names = OUT6 if mode == "forward" else OUT_INVERSE
    o = _properties(v if mode == "forward" else _temperature(v, p, Y, T), p, Y)
    return {**{k: torch.where(out, o[k], net[i]) for i, k in enumerate(names)}, "fallback": None}


def _rows(seed, batch, pool):
    """The pool rows of a batch: splitmix64 of the documented counter, modulo a power of two."""
    r = np.arange(batch, dtype=np.uint64)
    with np.errstate(over="ignore"):
        x = np.uint64(seed) ^ (r * np.uint64(0xD1B54A32D192ED03))
        x = x + np.uint64(0x9E3779B97F4A7C15)
        x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        x = x ^ (x >> np.uint64(31))
    return torch.as_tensor((x % np.uint64(pool)).astype(np.int64), device="cuda")


def _exact_train(case, seed):
    """The same Adam steps on the FP64 network (masked relative squared error)."""
    g = _generator(seed)
    x, y = _pool(case["mode"], case["pool"], g)
    layers, norm, _ = _model(case, x, y, g, False)
    nm = _col(norm, x)
    par = [v.double().clone().requires_grad_() for wb in layers for v in wb]
    m, s, losses = [torch.zeros_like(v) for v in par], [torch.zeros_like(v) for v in par], []
    for k in range(case["steps"]):
        rows = _rows(k + 1, case["batch"], case["pool"])
        xb, yb = x[:, rows].double(), y[:, rows].double()
        f, t = _features(case["mode"], xb[0], xb[1], xb[2:]), _targets(case["mode"], xb[0], xb[2:], yb)
        f = ((f - nm[:13, None]) / nm[13:26, None]).T
        t = ((t - nm[26:32, None]) / nm[32:38, None]).T
        pred = _forward([(par[2 * i], par[2 * i + 1]) for i in range(len(par) // 2)], f)
        fine = torch.isfinite(t)
        d = torch.where(fine, pred - torch.where(fine, t, torch.zeros_like(t)), torch.zeros_like(t))
        loss = (d * d).sum() / t.numel()
        grads = torch.autograd.grad(loss, par)
        losses.append(loss.detach())
        with torch.no_grad():
            for i, gr in enumerate(grads):
                m[i] = 0.9 * m[i] + 0.1 * gr
                s[i] = 0.999 * s[i] + 0.001 * gr * gr
                par[i] -= 1e-3 * (m[i] / (1 - 0.9 ** (k + 1))) / ((s[i] / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    return {"loss": torch.stack(losses), "params": torch.cat([v.detach().reshape(-1) for v in par]).cpu().numpy()}
