"""The work this package is measured on: what its users have it do, through its public entry points.

A molecular-dynamics program with a hybrid functional calls the exact exchange (E_x and V_x phi over a
pair list) on its slow steps, the ACE operator on its fast ones, the localisation and the overlap screen
when it renews its pair list, and the thermostat updates on every step.  The listed cases are those
calls at the sizes of this repository's workloads (orbitals and grids of water boxes, 16 orbitals on
32^3 to 256 on 96^3, a 128^3 grid) and at sizes off them: orbital counts that are no multiple of a
block, grids that are neither cubic nor a tuned edge, both precisions, orbitals held in either type.

Result types: a double-precision context's results are kept in double.  A single-precision context
computes in single precision and hands back its results in double arrays; the program here keeps them in
single precision, which is what they hold (the repository states them to 1e-7).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2309_00651_gb300 import hfx
from paper_2309_00651_gb300.autograd import exchange_energy
from paper_2309_00651_gb300.sinr import SinR

ALPHA = 0.25
WATER_BOHR3 = 202.4  # volume of one H2O, four doubly occupied orbitals, in liquid water


def _exchange(name, grid, n_orb, box, prec="fp32", orb="f64", kind="pw", ecut=20.0, sigma=1.2, keep=1.0, **more):
    c = {"do": "exchange", "n1": grid[0], "n2": grid[1], "n3": grid[2], "orbitals": n_orb, "L1": box[0], "L2": box[1],
         "L3": box[2], "precision": prec, "orb_type": orb, "kind": kind, "ecut": ecut, "sigma": sigma, "keep": keep}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest system a caller has: 16 orbitals, 136 pairs on 32^3; a call is mostly launches
        _exchange("exchange_o16_n32", (32, 32, 32), 16, (10.0,) * 3),
        # 32 H2O, every pair: the repository's headline workload
        _exchange("exchange_o128_n72", (72, 72, 72), 128, (18.6,) * 3, kind="gauss", ecut=40.0),
        # 64 H2O, every pair: the largest dense call
        _exchange("exchange_o256_n96", (96, 96, 96), 256, (23.5,) * 3),
        # a box of the uneven batch (80^3) with an orbital count that leaves a ragged block; a program
        # that holds its orbitals in single precision
        _exchange("exchange_o117_n80_f32orb", (80, 80, 80), 117, (19.8,) * 3, orb="f32"),
        # an orthorhombic cell with three different edges, none of them a tuned cube
        _exchange("exchange_o27_n54x60x72", (54, 60, 72), 27, (13.5, 15.0, 18.0)),
        # localised orbitals in a large box: the overlap-screened list, which leaves holes in most blocks
        _exchange("exchange_screened_o96_n128", (128, 128, 128), 96, (29.6,) * 3, kind="gauss", ecut=40.0, sigma=1.5, keep=0.35),
        # double precision throughout: reference runs and tight convergence
        _exchange("exchange_o24_n48_fp64", (48, 48, 48), 24, (12.0,) * 3, prec="fp64"),
        # a gradient step of an optimiser: E_x forward without storing V_x phi, its adjoint backward
        _exchange("gradient_o64_n64_f32orb", (64, 64, 64), 64, (15.0,) * 3, orb="f32", do="gradient"),
        # independent small boxes of different sizes in one batched call
        {"name": "batch_6_o24_n32_to_o72_n64", "do": "batch", "problems": 6, "lo": 24, "hi": 72},
        # the fast steps: ACE built from orbitals and V_x phi, then applied to them
        {"name": "ace_o128_n72", "do": "ace", "n1": 72, "n2": 72, "n3": 72, "orbitals": 128, "L1": 18.6, "L2": 18.6,
         "L3": 18.6, "precision": "fp32", "kind": "gauss", "ecut": 40.0, "sigma": 1.2},
        # renewing the pair list: localise the orbitals, then screen their overlaps
        {"name": "localise_o128_n72", "do": "localise", "n1": 72, "n2": 72, "n3": 72, "orbitals": 128, "L1": 18.6,
         "L2": 18.6, "L3": 18.6, "precision": "fp32", "kind": "gauss", "ecut": 40.0, "sigma": 1.2},
        # one outer step of the integrator for 128 H2O (1152 degrees of freedom), four inner steps
        {"name": "integrator_1152", "do": "integrator", "dof": 1152, "chain": 4, "n_mts": 4, "n_sy": 3},
    ]


CUBES = (24, 30, 32, 36, 40, 48, 50, 54, 60, 64, 72, 80, 90, 96, 108, 120, 128)
MOST_WORK = 32896 * 96.0 ** 3 / 4  # pairs x grid points of a drawn exchange call


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _orbital_cap(box, kind, points):
    """Most orbitals of a box: Gaussians at liquid-water density, plane waves well inside their sphere."""
    volume = box[0] * box[1] * box[2]
    dense = 4 * volume / WATER_BOHR3
    return max(4, int(min(256, dense if kind == "gauss" else 1.5 * dense, math.sqrt(2 * MOST_WORK / points))))


def draw(rng):
    do = rng.choice(["exchange"] * 7 + ["gradient", "gradient", "batch", "ace", "localise", "integrator"])
    if do == "batch":
        lo = rng.randint(8, 40)
        return {"do": do, "problems": rng.randint(2, 8), "lo": lo, "hi": lo + rng.randint(1, 60)}
    if do == "integrator":
        return {"do": do, "dof": 3 * _log(rng, 32, 400000), "chain": rng.randint(1, 6), "n_mts": rng.randint(1, 6),
                "n_sy": rng.choice([1, 3, 5])}
    if do in ("ace", "localise"):
        n = rng.choice([n for n in CUBES if 32 <= n <= 80])
        L = n / 3.9
        return {"do": do, "n1": n, "n2": n, "n3": n, "orbitals": _log(rng, 8, max(9, 4 * L ** 3 / WATER_BOHR3)), "L1": L,
                "L2": L, "L3": L, "precision": "fp32", "kind": "gauss", "ecut": 20.0, "sigma": 1.2}
    prec = rng.choice(["fp32"] * 6 + ["fp64"])
    kind = rng.choice(["pw", "gauss"])
    if prec == "fp64":
        grid = (rng.choice([n for n in CUBES if n <= 64]),) * 3
    elif rng.random() < 0.25:
        grid = tuple(rng.choice([n for n in CUBES if 30 <= n <= 96]) for _ in range(3))
    else:
        grid = (rng.choice(CUBES[2:]),) * 3
    box = tuple(n / 4.0 for n in grid)
    points = grid[0] * grid[1] * grid[2]
    n_orb = _log(rng, 4, _orbital_cap(box, kind, points))
    if prec == "fp64":
        n_orb = min(n_orb, 40)
    keep = 1.0 if rng.random() < 0.6 else rng.uniform(0.2, 0.9)
    orb = "f32" if do == "gradient" or rng.random() < 0.4 else "f64"
    if do == "gradient" or orb == "f32":
        prec = "fp32"
    return _exchange(None, grid, n_orb, box, prec=prec, orb=orb, kind=kind, keep=keep, do=do)


# ------------------------------------------------------------------------------------------------
# inputs, from the seed alone
# ------------------------------------------------------------------------------------------------

def _half_g(grid, box):
    """(G components on the half grid of a real transform, |G|^2)."""
    g1 = 2 * math.pi / box[0] * torch.fft.fftfreq(grid[0], 1.0 / grid[0], dtype=torch.float64, device="cuda")
    g2 = 2 * math.pi / box[1] * torch.fft.fftfreq(grid[1], 1.0 / grid[1], dtype=torch.float64, device="cuda")
    g3 = 2 * math.pi / box[2] * torch.fft.rfftfreq(grid[2], 1.0 / grid[2], dtype=torch.float64, device="cuda")
    return (g1, g2, g3), g1[:, None, None] ** 2 + g2[None, :, None] ** 2 + g3[None, None, :] ** 2


def _orbitals(grid, box, n_orb, kind, ecut, sigma, seed):
    """Orthonormal real orbitals [n_orb, n1, n2, n3] in double: damped random plane waves, or Gaussians
    around jittered molecule sites (four a molecule)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    (g1, g2, g3), gg = _half_g(grid, box)
    sphere = 0.5 * gg < ecut
    phi = torch.empty((n_orb,) + tuple(grid), dtype=torch.float64, device="cuda")
    if kind == "pw":
        amp = torch.exp(-gg / 8.0) * sphere
        for i in range(n_orb):
            c = torch.randn(amp.shape + (2,), dtype=torch.float64, device="cuda", generator=gen)
            phi[i] = torch.fft.irfftn(torch.view_as_complex(c) * amp, s=grid, norm="forward")
    else:
        rng = np.random.default_rng(seed)
        molecules = (n_orb + 3) // 4
        m = math.ceil(molecules ** (1.0 / 3.0) - 1e-12)
        cells = rng.permutation(m ** 3)[:molecules]
        sites = (np.stack([cells // (m * m), cells // m % m, cells % m], 1) + 0.5 + rng.uniform(-0.25, 0.25, (molecules, 3))) / m
        corners = np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]]) / math.sqrt(3.0)
        centres = (sites[:, None, :] * np.array(box) + 0.7 * corners).reshape(-1, 3)[:n_orb]
        amp = torch.exp(-0.5 * sigma * sigma * gg) * sphere
        for i, c in enumerate(centres):
            e = [torch.exp(-1j * g * float(x)) for g, x in zip((g1, g2, g3), c)]
            phi[i] = torch.fft.irfftn(amp * e[0][:, None, None] * e[1][None, :, None] * e[2][None, None, :], s=grid, norm="forward")
    flat = phi.reshape(n_orb, -1)
    weight = box[0] * box[1] * box[2] / flat.shape[1]
    w, u = torch.linalg.eigh(weight * (flat @ flat.T))
    return ((u * w.rsqrt()) @ u.T @ flat).reshape(phi.shape)


def _pair_count(n_orb, keep):
    full = n_orb * (n_orb + 1) // 2
    return full if keep >= 1.0 else max(n_orb, int(keep * full))


def _pairs(phi, keep):
    """Every pair i <= j, or the share `keep` of them with the largest overlaps (the diagonal always)."""
    n = phi.shape[0]
    ij = torch.triu_indices(n, n, device="cuda")
    if keep < 1.0:
        a = phi.reshape(n, -1).abs()
        s = (a @ a.T)[ij[0], ij[1]]
        s[ij[0] == ij[1]] = math.inf
        kept = torch.sort(torch.topk(s, _pair_count(n, keep)).indices).values
        ij = ij[:, kept]
    return ij.T.to(torch.int32).contiguous()


def _grid_box(case):
    return (case["n1"], case["n2"], case["n3"]), (case["L1"], case["L2"], case["L3"])


def _context(grid, box, precision):
    return hfx.Exchange(np.diag(box).tolist(), grid, alpha=ALPHA, precision=precision)


def _exchange_inputs(case, seed):
    grid, box = _grid_box(case)
    phi = _orbitals(grid, box, case["orbitals"], case["kind"], case["ecut"], case["sigma"], seed)
    pairs = _pairs(phi, case["keep"])
    return phi.to(torch.float32) if case["orb_type"] == "f32" else phi, pairs


def _batch_problems(case):
    """(orbitals, grid edge, box edge) of each box of a batch: orbital counts spread evenly from lo to
    hi, boxes at liquid-water density, the grid the smallest even {2,3,5}-smooth one of 4.03 points a bohr."""
    out = []
    for k in range(case["problems"]):
        n_orb = case["lo"] + (case["hi"] - case["lo"]) * k // max(1, case["problems"] - 1)
        L = (WATER_BOHR3 * n_orb / 4) ** (1.0 / 3.0)
        out.append((n_orb, min(n for n in CUBES if n >= 4.03 * L), L))
    return out


def _ace_inputs(case, seed):
    """Orbitals and W = a negative definite screened-Coulomb operator on them, as V_x phi is."""
    grid, box = _grid_box(case)
    phi = _orbitals(grid, box, case["orbitals"], case["kind"], case["ecut"], case["sigma"], seed)
    _, gg = _half_g(grid, box)
    w = torch.empty_like(phi)
    for i in range(phi.shape[0]):
        w[i] = torch.fft.irfftn(torch.fft.rfftn(phi[i]) * (-4 * math.pi / (gg + 4.0)), s=grid)
    return phi, w


KT, TAU, DT = 300 * 3.166811563e-6, 413.0, 20.67  # 300 K, 10 fs, 0.5 fs in atomic units


def _integrator_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, L = case["dof"], case["chain"]

    def normal(*shape):
        return torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)

    atom = torch.arange(n, device="cuda") // 3
    mass = torch.where(atom % 3 == 0, 29156.9, 1837.4).to(torch.float64)
    q = KT * TAU * TAU
    X, V, v1, v2 = 0.1 * normal(n), normal(n) * (KT / mass).sqrt(), normal(n, L) * math.sqrt(KT / q), normal(n, L) * math.sqrt(KT / q)
    lam = mass * V * V + L / (L + 1.0) * q * (v1 * v1).sum(-1)  # the constraint the updates keep: L kT
    scale = (L * KT / lam).sqrt()
    return gen, X, V * scale, v1 * scale[:, None], v2, mass, q


def _fast(X):
    return -0.3 * X


def _slow(X):
    return -0.02 * X


def prepare(case, seed):
    do = case["do"]
    s = {"do": do}
    if do in ("exchange", "gradient"):
        s["phi"], s["pairs"] = _exchange_inputs(case, seed)
        s["ctx"] = _context(*_grid_box(case), case["precision"])
        s["keep_as"] = torch.float64 if case["precision"] == "fp64" else torch.float32
        if do == "gradient":
            s["phi"].requires_grad_(True)
    elif do == "batch":
        s["ctxs"], s["args"] = [], []
        for k, (n_orb, n, L) in enumerate(_batch_problems(case)):
            phi = _orbitals((n,) * 3, (L,) * 3, n_orb, "pw", 20.0, 0.0, seed * 64 + k)
            ctx, pairs = _context((n,) * 3, (L,) * 3, "fp32"), _pairs(phi, 1.0)
            ctx.ensure_workspace(n_orb, pairs.shape[0])
            s["ctxs"].append(ctx)
            s["args"].append((phi, pairs, torch.zeros(1, dtype=torch.float64, device="cuda"), torch.empty_like(phi), 0))
    elif do == "ace":
        s["phi"], s["w"] = _ace_inputs(case, seed)
        s["ctx"] = _context(*_grid_box(case), case["precision"])
    elif do == "localise":
        grid, box = _grid_box(case)
        s["phi"] = _orbitals(grid, box, case["orbitals"], case["kind"], case["ecut"], case["sigma"], seed)
        s["ctx"] = _context(grid, box, case["precision"])
    else:
        s["gen"], s["X"], s["V"], s["v1"], s["v2"], s["mass"], q = _integrator_inputs(case, seed)
        s["step"] = SinR(KT, q, q, 1.0 / 8000.0, case["chain"], n_sy=case["n_sy"])
        s["n_mts"] = case["n_mts"]
    return s


def run(s):
    do = s["do"]
    if do == "exchange":
        E, V = s["ctx"].apply(s["phi"], s["pairs"])
        return {"E": E.to(s["keep_as"]), "V": V.to(s["keep_as"])}
    if do == "gradient":
        E = exchange_energy(s["ctx"], s["phi"], s["pairs"], recompute=True)
        (grad,) = torch.autograd.grad(E, s["phi"])
        return {"E": E.detach().to(s["keep_as"]), "grad": grad}
    if do == "batch":
        hfx.hfx_apply_batched([c.ctx for c in s["ctxs"]], s["args"])
        return [{"E": a[2].float(), "V": a[3].float()} for a in s["args"]]
    if do == "ace":
        m, l, p = s["ctx"].ace_build(s["phi"], s["w"])
        out = s["ctx"].ace_apply(p, s["phi"])
        return {"M": m.float(), "L": l.float(), "P": p.float(), "V": out.float()}
    if do == "localise":
        pivots, q, phi = s["ctx"].scdm_localise(s["phi"])
        pairs, overlaps = s["ctx"].screen_pairs(phi, 1e-3)
        near = torch.zeros(overlaps.shape, dtype=torch.bool, device=phi.device)  # the program's neighbour table
        near[pairs[:, 0].long(), pairs[:, 1].long()] = True
        return {"pivots": pivots, "q": q.float(), "phi": phi.float(), "near": near, "s": overlaps.float()}
    shape = s["v2"].shape
    s["step"].outer(s["X"], s["V"], s["v1"], s["v2"], s["mass"], _fast, _slow, DT, s["n_mts"],
                    lambda: torch.randn(shape, dtype=torch.float64, device="cuda", generator=s["gen"]))
    return {"X": s["X"], "V": s["V"], "v1": s["v1"], "v2": s["v2"]}


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------

def _exchange_work(points, n_orb, n_pairs, in_bytes, out_bytes, energy_only=False):
    """Inputs read and outputs written once; per pair a forward and an inverse real transform of
    2.5 N log2 N each, the pair product, the Coulomb multiply with its energy, and two accumulations."""
    flops = n_pairs * points * ((2.5 if energy_only else 5.0) * math.log2(points) + (6 if energy_only else 10))
    return {"bytes": points * n_orb * (in_bytes + out_bytes), "flops": flops}


def work(case):
    do = case["do"]
    if do == "batch":
        parts = [_exchange_work(n ** 3, m, m * (m + 1) // 2, 8, 4) for m, n, _ in _batch_problems(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if do == "integrator":
        state = case["dof"] * 8 * (2 * (2 + 2 * case["chain"]) + 1)
        return {"bytes": state, "flops": case["dof"] * case["n_mts"] * (2 * case["n_sy"] * (40 * case["chain"] + 10) + 120)}
    points, n = case["n1"] * case["n2"] * case["n3"], case["orbitals"]
    if do == "ace":  # phi, W in; P and V_x^ACE phi out; four contractions
        return {"bytes": points * n * (8 + 8 + 4 + 4), "flops": 4 * 2.0 * n * n * points}
    if do == "localise":  # phi in, phi out; the pivoting's n sweeps of n-term products, Psi Q, the overlaps
        return {"bytes": points * n * (8 + 4), "flops": 3 * 2.0 * n * n * points}
    size = 4 if case["orb_type"] == "f32" else 8
    keep = 8 if case["precision"] == "fp64" else 4
    n_pairs = _pair_count(n, case["keep"])
    w = _exchange_work(points, n, n_pairs, size, keep)
    if do == "gradient":
        w["flops"] += _exchange_work(points, n, n_pairs, size, 0, energy_only=True)["flops"]
    return w


# ------------------------------------------------------------------------------------------------
# the same in 64 bits, plainly
# ------------------------------------------------------------------------------------------------

def _exact_exchange(phi, pairs, grid, box):
    phi = phi.detach().to(torch.float64)
    n, points = phi.shape[0], grid[0] * grid[1] * grid[2]
    volume = box[0] * box[1] * box[2]
    _, gg = _half_g(grid, box)
    v = torch.where(gg > 0, 4 * math.pi / gg.clamp_min(1e-300), torch.zeros_like(gg))
    both = torch.full_like(v, 2.0)  # a half-grid point stands for G and -G, except on the planes that are their own mirror
    both[..., 0] = 1.0
    if grid[2] % 2 == 0:
        both[..., -1] = 1.0
    E, V = torch.zeros((), dtype=torch.float64, device="cuda"), torch.zeros_like(phi)
    by_first = {}
    for i, j in pairs.tolist():
        by_first.setdefault(i, []).append(j)
    chunk = max(1, int(3e7 / points))
    for i, js in by_first.items():
        for k in range(0, len(js), chunk):
            j = torch.tensor(js[k:k + chunk], device="cuda")
            F = torch.fft.rfftn(phi[i] * phi[j], dim=(1, 2, 3))
            weight = torch.where(j == i, 1.0, 2.0).to(torch.float64)
            E += (weight * (v * both * (F.real ** 2 + F.imag ** 2)).sum(dim=(1, 2, 3))).sum()
            pot = torch.fft.irfftn(v * F, s=grid, dim=(1, 2, 3))
            V[i] -= ALPHA * torch.einsum("jxyz,jxyz->xyz", pot, phi[j])
            off = j != i
            V[j[off]] -= ALPHA * pot[off] * phi[i]
    return (-0.5 * ALPHA * volume / points ** 2 * E).reshape(1), V


def _exact_integrator(case, seed):
    gen, X, V, v1, v2, M, q = _integrator_inputs(case, seed)
    L, gamma, lam, h = case["chain"], 1.0 / 8000.0, case["chain"] * KT, 0.5 * DT
    if case["n_sy"] == 1:
        weights = [1.0]
    else:
        k = case["n_sy"] - 1
        w = 1.0 / (k - k ** (1.0 / 3.0))
        weights = [w] * (k // 2) + [1.0 - k * w] + [w] * (k // 2)

    def thermostat(V, v1, v2):
        for w in weights:
            d = w * DT
            v2 = v2 + 0.25 * d * (q * v1 * v1 - KT) / q
            H = (lam / (M * V * V + L / (L + 1.0) * q * (v1 * v1 * torch.exp(-v2 * d)).sum(-1))).sqrt()
            V, v1 = V * H, v1 * H[:, None] * torch.exp(-0.5 * v2 * d)
            v2 = v2 + 0.25 * d * (q * v1 * v1 - KT) / q
        return V, v1, v2

    def kick(V, v1, F):
        a, b = F * V / lam, F * F / (M * lam)
        x = b.sqrt() * h
        small = x < 1e-4
        c = torch.where(small, torch.ones_like(b), b)
        s = torch.where(small, h * (1 + x * x / 6) + a * h * h * (0.5 + x * x / 24), torch.sinh(x) / c.sqrt() + a / c * 2 * torch.sinh(0.5 * x) ** 2)
        sd = torch.where(small, 1 + x * x / 2 + a * h * (1 + x * x / 6), torch.cosh(x) + a / c.sqrt() * torch.sinh(x))
        return (V + s * F / M) / sd, v1 / sd[:, None]

    for k in range(case["n_mts"]):
        V, v1, v2 = thermostat(V, v1, v2)
        V, v1 = kick(V, v1, _fast(X) + (case["n_mts"] * _slow(X) if k == 0 else 0.0))
        R = torch.randn(v2.shape, dtype=torch.float64, device="cuda", generator=gen)
        X = X + V * DT
        v2 = v2 * math.exp(-gamma * DT) + math.sqrt(KT / q * (1.0 - math.exp(-2.0 * gamma * DT))) * R
        V, v1 = kick(V, v1, _fast(X) + (case["n_mts"] * _slow(X) if k == case["n_mts"] - 1 else 0.0))
        V, v1, v2 = thermostat(V, v1, v2)
    return {"X": X, "V": V, "v1": v1, "v2": v2}


def exact(case, seed):
    do = case["do"]
    if do == "exchange":
        phi, pairs = _exchange_inputs(case, seed)
        E, V = _exact_exchange(phi, pairs, *_grid_box(case))
        return {"E": E, "V": V}
    if do == "gradient":
        phi, pairs = _exchange_inputs(case, seed)
        E, V = _exact_exchange(phi, pairs, *_grid_box(case))
        grid, box = _grid_box(case)
        return {"E": E.reshape(()), "grad": 2 * box[0] * box[1] * box[2] / (grid[0] * grid[1] * grid[2]) * V}
    if do == "batch":
        out = []
        for k, (n_orb, n, L) in enumerate(_batch_problems(case)):
            phi = _orbitals((n,) * 3, (L,) * 3, n_orb, "pw", 20.0, 0.0, seed * 64 + k)
            E, V = _exact_exchange(phi, _pairs(phi, 1.0), (n,) * 3, (L,) * 3)
            out.append({"E": E, "V": V})
        return out
    if do == "integrator":
        return _exact_integrator(case, seed)
    grid, box = _grid_box(case)
    weight = box[0] * box[1] * box[2] / (grid[0] * grid[1] * grid[2])
    if do == "ace":
        phi, w = _ace_inputs(case, seed)
        f, g = phi.reshape(phi.shape[0], -1), w.reshape(w.shape[0], -1)
        M = weight * (f @ g.T)
        L = torch.linalg.cholesky(-0.5 * (M + M.T))
        P = torch.linalg.solve_triangular(L, g, upper=False)
        V = -(weight * (f @ P.T)) @ P
        return {"M": M, "L": L, "P": P.reshape(phi.shape), "V": V.reshape(phi.shape)}
    # greedy column-pivoted QR of Psi^T; the picks themselves are whole numbers and have no 64-bit value
    phi = _orbitals(grid, box, case["orbitals"], case["kind"], case["ecut"], case["sigma"], seed)
    n = phi.shape[0]
    A, Q = phi.reshape(n, -1), []
    nu = (A * A).sum(0)
    for _ in range(n):
        p = int(torch.argmax(nu))
        r = A[:, p].clone()
        for _ in range(2):
            for u in Q:
                r = r - u * (u @ r)
        Q.append(r / r.norm())
        nu = nu - (Q[-1] @ A) ** 2
        nu[p] = -1.0
    Q = torch.stack(Q, 1)
    loc = Q.T @ A
    a = loc.abs()
    return {"pivots": None, "q": Q, "phi": loc.reshape(phi.shape), "near": None, "s": weight * (a @ a.T)}
