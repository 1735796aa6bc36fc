"""The calls whose time matters to a user of this library, with their inputs.

A case is one call, or the few calls that a program always makes together, on
one cell.  The sizes are those of the workloads in
``paper_1611_00731_gb300/workloads.py`` and of the tests, from the 8-element
cells of an equation-of-state sweep to the 64-atom supercell.

``call`` says what a pass does:
  step      what one iteration of a solver needs of the library: the
            enrichment table, H and S, the density and the derivative with
            respect to the potential (at a wavevector if ``bloch``)
  grad      H(V) and its vector-Jacobian product through torch.autograd
  scf       H and S of the input potential, then one self-consistent step
            (occupations, density, energies, mixing, the new potential)
  kpoint    H(k), S(k) and the density of the complex states of one k-point
  project   the projections of the basis onto nonlocal projectors
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1611_00731_gb300 import autograd, pufe, workloads as W

F64 = torch.float64
KT = 0.01   # hartree, the smearing of the self-consistent steps


def listed():
    return [
        # one cell of an equation-of-state sweep: 8 elements, 6^3 points each, in
        # the default precision; launches and waits are all of its time
        dict(name="eos_scf_fp64", cell="two_atom", nel=2, p=6, prec="fp64", call="scf", nocc=6),
        # the two-atom Gamma-point cell (4^3 elements, 8^3 points near the atoms)
        dict(name="two_atom_step_fp64", cell="two_atom", nel=4, p=8, prec="fp64", call="step",
             nocc=2),
        # the rocksalt cube, 12^3 elements: the workload of the benchmark, in both
        # precisions, and its self-consistent iteration
        dict(name="rocksalt_step_mixed", cell="rocksalt", nel=12, prec="mixed", call="step",
             nocc=8),
        dict(name="rocksalt_step_fp64", cell="rocksalt", nel=12, prec="fp64", call="step", nocc=8),
        dict(name="rocksalt_scf_mixed", cell="rocksalt", nel=12, prec="mixed", call="scf", nocc=12),
        # differentiation on a mesh too fine to keep the basis: forward and backward
        dict(name="rocksalt_grad_mixed", cell="rocksalt", nel=20, prec="mixed", call="grad",
             nocc=8),
        # one k-point of a coarser rocksalt cube, 9^3 elements, in the default precision
        dict(name="rocksalt_bloch_fp64", cell="rocksalt", nel=9, prec="fp64", call="step", nocc=8,
             bloch=True),
        # s and p projectors on each of the eight atoms
        dict(name="rocksalt_project", cell="rocksalt", nel=12, prec="fp64", call="project",
             nocc=1),
        # CsCl-type cell: eight elements of 184 functions and 4096 points among 4,032
        # plain ones of 64 and 64; odd number of states
        dict(name="cscl_step_mixed", cell="cscl", nel=16, prec="mixed", call="step", nocc=35),
        dict(name="cscl_step_fp64", cell="cscl", nel=16, prec="fp64", call="step", nocc=35),
        # 64 atoms, 32^3 elements: one of the four k-points, 64 complex states
        dict(name="supercell_kpoint_mixed", cell="supercell", nel=16, prec="mixed", call="kpoint",
             nocc=64, bloch=True),
        # triclinic cell with the serendipity elements, at a wavevector
        dict(name="triclinic_bloch_fp64", cell="triclinic", nel=6, p=6, fe="serendipity32",
             prec="fp64", call="step", nocc=4, bloch=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    cell = rng.choice(["two_atom", "two_atom", "rocksalt", "rocksalt", "rocksalt", "cscl",
                       "supercell", "triclinic"])
    prec = rng.choice(["fp64", "mixed"])
    if cell == "two_atom":
        return dict(cell=cell, nel=rng.randint(2, 6), p=rng.randint(4, 9), prec=prec,
                    call=rng.choice(["step", "grad", "scf", "project"]), nocc=_log(rng, 2, 64))
    if cell == "rocksalt":
        call = rng.choice(["step", "step", "grad", "scf", "kpoint", "project"])
        return dict(cell=cell, nel=rng.randint(4, 14), prec=prec, call=call,
                    nocc=_log(rng, 8, 64), bloch=call == "kpoint" or (
                        call in ("step", "project") and rng.random() < 0.4))
    if cell == "cscl":
        return dict(cell=cell, nel=rng.randint(6, 16), prec=prec,
                    call=rng.choice(["step", "grad"]), nocc=_log(rng, 8, 40))
    if cell == "supercell":
        return dict(cell=cell, nel=rng.randint(4, 12), prec="mixed", call="kpoint",
                    nocc=rng.randint(33, 64), bloch=True)
    call = rng.choice(["step", "step", "grad"])
    return dict(cell=cell, nel=rng.randint(2, 7), p=rng.randint(4, 8),
                fe=rng.choice(["lagrange64", "serendipity32"]), prec="fp64", call=call,
                nocc=_log(rng, 1, 16), bloch=call == "step" and rng.random() < 0.5)


# --- the cells and what a program holds before the call ------------------------


def _cell(case):
    if case["cell"] == "two_atom":
        wl = W.workload("c1_two_atom_4cube")
        if case["call"] == "scf":   # the cells of the equation-of-state sweep
            wl = W.small_two_atom(nel=case["nel"], a=6.15, quad_p=case["p"])
        else:
            wl["nel"] = case["nel"]
            wl["quad"] = dict(wl["quad"], p_near=case["p"])
        return wl
    if case["cell"] == "rocksalt":
        return W.workload("c2_rocksalt_%dcube" % case["nel"])
    if case["cell"] == "cscl":
        return W.workload("c3_cscl_%dcube" % case["nel"])
    if case["cell"] == "supercell":
        return W.workload("c5_rocksalt_2x2x2_%dcube" % case["nel"])
    wl = W.ceal_like(nel=case["nel"], quad_p=case["p"])
    wl["fe"] = case["fe"]
    return wl


def _prec(case):
    return pufe.PUFE_FP64 if case["prec"] == "fp64" else pufe.PUFE_TF32X3


def _lattice(wl):
    if wl.get("lattice") is not None:
        return np.array(wl["lattice"], dtype=np.float64)
    return np.eye(3) * float(wl["a"])


def _lattice_and_inverse(wl, dev):
    L = _lattice(wl)
    return torch.tensor(L, device=dev), torch.tensor(np.linalg.inv(L), device=dev)


def _wavevector(wl):
    """(1/4, 1/4, 1/4) in the reciprocal lattice."""
    return 2.0 * math.pi * np.linalg.solve(_lattice(wl), np.full(3, 0.25))


def _node_positions(wl):
    """Fractional coordinates of the FE nodes, in the order of their DOFs."""
    m = 3 * int(wl["nel"])
    g = np.arange(m ** 3)
    g3 = np.stack([g % m, (g // m) % m, g // (m * m)], axis=1)
    if wl.get("fe") == "serendipity32":
        g3 = g3[(g3 % 3 != 0).sum(axis=1) <= 1]
    return g3 / m


def _states(wl, n_dof, nocc, seed, dev, k=None):
    """Smooth states: three plane waves each on the FE nodes, small random
    enrichment coefficients; (re, im) at a wavevector, else real."""
    rs = np.random.RandomState(seed % (1 << 31))
    pos = torch.tensor(_node_positions(wl), device=dev)
    vol = abs(np.linalg.det(_lattice(wl)))
    gen = torch.Generator(device=dev).manual_seed(seed)
    kf = None if k is None else _lattice(wl) @ k / (2.0 * math.pi)
    re, im = torch.zeros(n_dof, nocc, dtype=F64, device=dev), None
    if k is not None:
        im = torch.zeros_like(re)
    amp = rs.normal(size=(3, nocc))
    amp /= np.sqrt((amp * amp).sum(axis=0))
    for j in range(3):
        G = rs.randint(-3, 4, size=(nocc, 3)) + 0.0
        G[(G == 0).all(axis=1)] = 1.0
        if kf is not None:
            G = G + kf
        th = 2.0 * math.pi * (pos @ torch.tensor(G.T, device=dev)
                              + torch.tensor(rs.uniform(size=nocc), device=dev))
        a = torch.tensor(amp[j], device=dev) / math.sqrt(vol)
        if k is None:
            re[:len(pos)] += math.sqrt(2.0) * a * torch.cos(th)
        else:
            re[:len(pos)] += a * torch.cos(th)
            im[:len(pos)] += a * torch.sin(th)
    for c in (re, im):
        if c is not None and n_dof > len(pos):
            c[len(pos):] = 0.05 * torch.randn(n_dof - len(pos), nocc, generator=gen, dtype=F64,
                                              device=dev)
    return re if k is None else (re, im)


def _potential(wl, x, seed):
    """The local potential -Z erf(r / sigma) / r of the nearest image of every
    atom, with a smooth modulation drawn from the seed."""
    L, inv = _lattice_and_inverse(wl, x.device)
    V = torch.zeros(len(x), dtype=F64, device=x.device)
    for s, tau in wl["atoms"]:
        sp = wl["species"][s]
        d = (x - torch.tensor(tau, dtype=F64, device=x.device)) @ inv
        r = torch.linalg.norm((d - torch.round(d)) @ L, dim=1).clamp_min(1e-12)
        V -= sp["Z"] * torch.erf(r / sp["sigma"]) / r
    rs = np.random.RandomState(seed % (1 << 31))
    frac = x @ inv
    for _ in range(4):
        G = torch.tensor(rs.randint(-2, 3, size=3) + 0.0, device=x.device)
        V *= 1.0 + 0.05 * torch.cos(2.0 * math.pi * (frac @ G + rs.uniform()))
        V += 0.1 * rs.uniform()
    return V


def _projectors(wl):
    out = []
    for _, tau in wl["atoms"]:
        out.append(dict(tau=tau, l=0, m=0, rp=0.8))
        out += [dict(tau=tau, l=1, m=m, rp=0.8) for m in (-1, 0, 1)]
    return out


def _cotangent(s, bloch):
    """sum_n f_n c_n c_n^* on the sparsity pattern: with it the derivative with
    respect to the potential is the density (Hellmann-Feynman)."""
    rowptr, col = s["ctx"].pattern()
    dev = s["f"].device
    rp = torch.tensor(rowptr, device=dev)
    row = torch.repeat_interleave(torch.arange(len(rp) - 1, device=dev), rp[1:] - rp[:-1])
    col = torch.tensor(col, device=dev).long()
    h = torch.zeros(len(col), dtype=F64, device=dev)
    hi = torch.zeros_like(h) if bloch else None
    for n in range(min(s["f"].numel(), 8)):
        cr = (s["C"][0] if bloch else s["C"])[:, n].contiguous()
        if not bloch:
            h += s["f"][n] * cr[row] * cr[col]
            continue
        ci = s["C"][1][:, n].contiguous()
        h += s["f"][n] * (cr[row] * cr[col] + ci[row] * ci[col])
        hi += s["f"][n] * (ci[row] * cr[col] - cr[row] * ci[col])
    return (h, hi) if bloch else h


def prepare(case, seed):
    wl = _cell(case)
    dev = torch.device("cuda", torch.cuda.current_device())
    prec, call = _prec(case), case["call"]
    bloch = bool(case.get("bloch"))
    ctx = pufe.pufe_build_mesh(wl)
    s = dict(ctx=ctx, wl=wl, prec=prec, call=call, bloch=bloch)
    new = lambda n: torch.empty(n, dtype=F64, device=dev)
    pair = (lambda n: (new(n), new(n))) if bloch else new
    if bloch:
        s["k"] = _wavevector(wl)
    if call != "step":   # a step tabulates by itself
        ctx.pufe_tabulate(pufe.PUFE_FP64 if call == "project" else prec)
    if call == "project":
        tau0 = np.random.RandomState(seed % (1 << 31)).uniform(-0.1, 0.1, size=3)
        s["proj"] = [dict(q, tau=tuple(np.asarray(q["tau"]) + tau0)) for q in _projectors(wl)]
        n = (ctx.n_dof, len(s["proj"]))
        s["F"] = pair(n)
        return s
    rs = np.random.RandomState(seed % (1 << 31))
    nocc = case["nocc"]
    s["C"] = _states(wl, ctx.n_dof, nocc, seed, dev, s.get("k"))
    s["f"] = torch.tensor(rs.uniform(0.0, 2.0, size=nocc), device=dev)
    x = torch.tensor(ctx.quadrature()[0], device=dev)
    if call == "scf":
        nelec = float(wl["nelec"])
        nst = max(nocc, int(nelec / 2) + 1)
        if nst != nocc:
            s["C"] = _states(wl, ctx.n_dof, nst, seed, dev)
        s["nelec"], s["eps"] = nelec, np.sort(rs.uniform(-0.6, 0.3, size=nst))
        at = [(tau, wl["species"][i]["Z"], wl["species"][i]["sigma"]) for i, tau in wl["atoms"]]
        s["atoms"] = tuple(np.array(v, dtype=np.float64) for v in zip(*at))
        s["rho_I"] = new(ctx.n_q)
        ctx.pufe_ion_density(*s["atoms"], s["rho_I"])
        G = torch.tensor(rs.randint(1, 3, size=3) + 0.0, device=dev)
        s["n_in"] = nelec / float(wl["a"]) ** 3 * (
            1.0 + 0.3 * torch.cos(2.0 * math.pi * (x @ G / float(wl["a"]) + rs.uniform())))
        s["n"], s["V"], s["V_out"] = new(ctx.n_q), new(ctx.n_q), new(ctx.n_q)
        ctx.pufe_effective_potential(s["n_in"], s["rho_I"], s["V"])
    else:
        s["V"] = _potential(wl, x, seed)
    if call == "grad":
        s["V"].requires_grad_(True)
    else:
        s["H"], s["S"] = pair(ctx.nnz), pair(ctx.nnz)
    if call in ("step", "kpoint"):
        s["rho"] = new(ctx.n_q)
    if call in ("step", "grad"):
        s["Hbar"], s["Vbar"] = _cotangent(s, bloch), new(ctx.n_q)
    return s


def run(s):
    ctx, prec = s["ctx"], s["prec"]
    if s["call"] == "project":
        if s["bloch"]:
            ctx.pufe_nonlocal_projections_bloch(s["k"], s["proj"], s["F"])
        else:
            ctx.pufe_nonlocal_projections(s["proj"], s["F"])
        return dict(F=s["F"])
    if s["call"] == "grad":
        H = autograd.assemble_H(ctx, s["V"], prec)
        return dict(H=H, V=torch.autograd.grad(H, s["V"], s["Hbar"])[0])
    if s["call"] == "scf":
        s["n"].copy_(s["n_in"])
        ctx.pufe_assemble_HS(s["V"], s["H"], s["S"], prec=prec)
        f, info = ctx.pufe_scf_step(s["eps"], s["C"], s["nelec"], KT, 0.5, s["rho_I"], s["V"],
                                    s["n"], s["V_out"], prec=prec)
        return dict(H=s["H"], S=s["S"], n=s["n"], V=s["V_out"], f=f, info=info)
    out = dict(H=s["H"], S=s["S"], rho=s["rho"])
    if s["call"] == "step":
        out["Vbar"] = s["Vbar"]
        ctx.pufe_tabulate(prec)
    if s["bloch"]:
        ctx.pufe_assemble_HS_bloch(s["k"], s["V"], s["H"], s["S"], prec=prec)
        ctx.pufe_density_bloch(s["k"], *s["C"], s["f"], s["rho"], prec=prec)
        if s["call"] == "step":
            ctx.pufe_assemble_HV_adjoint_bloch(s["k"], *s["Hbar"], s["Vbar"], prec=prec)
    else:
        ctx.pufe_assemble_HS(s["V"], s["H"], s["S"], prec=prec)
        ctx.pufe_density(s["C"], s["f"], s["rho"], prec=prec)
        if s["call"] == "step":
            ctx.pufe_assemble_HV_adjoint(s["Hbar"], s["Vbar"], prec=prec)
    return out


# --- bytes and operations of a pass ---------------------------------------------


@functools.lru_cache(maxsize=None)
def _sizes(key):
    ctx = pufe.pufe_build_mesh(_cell(dict(key)))
    _, _, off = ctx.quadrature()
    n_e, _ = ctx.element_basis()
    got = dict(n_q=ctx.n_q, n_dof=ctx.n_dof, nnz=ctx.nnz, Q=np.diff(off).astype(float),
               n=n_e.astype(float), A=ctx.element_slots().astype(float))
    ctx.close()
    return got


def work(case):
    """Each input read once, each output written once; the operations of the
    axis-by-axis contractions (two per multiply-add), the cheapest known
    forms of the integrals on tensor-product rules, with every element's rule
    taken as one p^3 grid."""
    z = _sizes(tuple(sorted(case.items())))
    c = 2 if case.get("bloch") else 1
    p, A, K = np.round(np.cbrt(z["Q"])), z["A"], case["nocc"]
    V, M, C = 8.0 * z["n_q"], 8.0 * z["nnz"] * c, 8.0 * z["n_dof"] * K * c
    rule, table = 32.0 * z["n_q"], float((z["Q"] * A).sum()) * (32.0 if case["prec"] == "fp64" else 16.0)
    pairs = A * (A + 1) / 2
    assemble = 2.0 * float((10 * p ** 3 + 100 * p ** 2 + 1000 * p
                            + A * (48 * p ** 3 + 320 * p ** 2 + 2048 * p)
                            + pairs * (59 * p ** 3 + 209 * p ** 2 + 597 * p)).sum())
    density = 2.0 * c * K * float((64 * p + 16 * p ** 2 + 4 * p ** 3
                                   + A * (8 * p + 4 * p ** 2 + 3 * p ** 3) + p ** 3).sum())
    adjoint = 2.0 * float((4096 * p + 256 * p ** 2 + 16 * p ** 3
                           + A * (512 * p + 64 * p ** 2 + 9 * p ** 3)
                           + pairs * (27 * p + 9 * p ** 2 + 4 * p ** 3)).sum())
    tabulate = 40.0 * float((z["Q"] * A).sum())
    call = case["call"]
    if call == "project":
        P = 4 * len(_cell(case)["atoms"])
        return dict(bytes=rule + table / 4 + 8.0 * z["n_dof"] * P * c,
                    flops=2.0 * c * P * float((p ** 3 + 4 * p ** 3 + 16 * p ** 2 + 64 * p
                                               + A * (3 * p ** 3 + 4 * p ** 2 + 8 * p)).sum()))
    if call == "grad":
        return dict(bytes=rule + table + 2 * V + 2 * M, flops=assemble + adjoint)
    if call == "scf":
        solve = 2.0 * 12.0 * (3 * case["nel"]) ** 4 + 300.0 * z["n_q"]
        return dict(bytes=rule + table + 4 * V + 2 * M + C, flops=assemble + density + solve)
    if call == "kpoint":
        return dict(bytes=rule + table + 2 * V + 2 * M + C, flops=assemble + density)
    return dict(bytes=rule + table + 3 * V + 3 * M + C,
                flops=tabulate + assemble + density + adjoint)


# --- the same results in 64 bits -------------------------------------------------
# The rule, every element's columns and the sparsity pattern are the plan's (points
# and whole numbers that the calls take as given); every number is formed here.

_C0, _C1 = 0.5 / math.sqrt(math.pi), math.sqrt(3.0 / (4.0 * math.pi))
_C2, _C20 = math.sqrt(15.0 / math.pi) / 2.0, math.sqrt(5.0 / math.pi) / 4.0
_C3, _C32 = math.sqrt(35.0 / (2.0 * math.pi)) / 4.0, math.sqrt(105.0 / math.pi) / 2.0
_C31, _C30 = math.sqrt(21.0 / (2.0 * math.pi)) / 4.0, math.sqrt(7.0 / math.pi) / 4.0
# r^l Y_lm as sums of monomials (powers of x, y, z)
_SOLID = {
    (0, 0): {(0, 0, 0): _C0},
    (1, -1): {(0, 1, 0): _C1}, (1, 0): {(0, 0, 1): _C1}, (1, 1): {(1, 0, 0): _C1},
    (2, -2): {(1, 1, 0): _C2}, (2, -1): {(0, 1, 1): _C2}, (2, 1): {(1, 0, 1): _C2},
    (2, 0): {(0, 0, 2): 2 * _C20, (2, 0, 0): -_C20, (0, 2, 0): -_C20},
    (2, 2): {(2, 0, 0): _C2 / 2, (0, 2, 0): -_C2 / 2},
    (3, -3): {(2, 1, 0): 3 * _C3, (0, 3, 0): -_C3}, (3, -2): {(1, 1, 1): _C32},
    (3, -1): {(0, 1, 2): 4 * _C31, (2, 1, 0): -_C31, (0, 3, 0): -_C31},
    (3, 0): {(0, 0, 3): 2 * _C30, (2, 0, 1): -3 * _C30, (0, 2, 1): -3 * _C30},
    (3, 1): {(1, 0, 2): 4 * _C31, (3, 0, 0): -_C31, (1, 2, 0): -_C31},
    (3, 2): {(2, 0, 1): _C32 / 2, (0, 2, 1): -_C32 / 2},
    (3, 3): {(3, 0, 0): _C3, (1, 2, 0): -3 * _C3},
}


def _solid(l, m, d):
    """r^l Y_lm and its gradient at the displacements d (..., 3)."""
    v = torch.zeros_like(d[..., 0])
    g = [torch.zeros_like(v) for _ in range(3)]
    for pw, c in _SOLID[(l, m)].items():
        t = [d[..., i] ** pw[i] for i in range(3)]
        v = v + c * t[0] * t[1] * t[2]
        for i in range(3):
            if pw[i]:
                o = [t[j] if j != i else pw[i] * d[..., i] ** (pw[i] - 1) for j in range(3)]
                g[i] = g[i] + c * o[0] * o[1] * o[2]
    return v, g


def _images(wl, reach, dev):
    """Lattice vectors that can bring a point's nearest image, or any other
    within `reach`, into play."""
    L = _lattice(wl)
    if wl.get("lattice") is None and reach <= float(wl["a"]) / 2:
        return torch.zeros(1, 3, dtype=F64, device=dev)
    h = 1.0 / np.linalg.norm(np.linalg.inv(L), axis=0)   # distance of the lattice planes
    n = [int(math.ceil(reach / float(v) + 0.5)) for v in h]
    ijk = np.stack(np.meshgrid(*[np.arange(-v, v + 1) for v in n], indexing="ij"), -1)
    return torch.tensor(ijk.reshape(-1, 3) @ L, device=dev)


def _orbital(wl, orb, rc, d):
    """Psi and grad Psi of one orbital at displacements d (..., 3) from its atom."""
    n, l, m, zeta = orb
    L, inv = _lattice_and_inverse(wl, d.device)
    d = d - torch.round(d @ inv) @ L
    norm = (2.0 * zeta) ** (n + 0.5) / math.sqrt(math.factorial(2 * n))
    out = [torch.zeros_like(d[..., 0]) for _ in range(4)]
    for R in _images(wl, rc, d.device):
        e = d + R
        r = torch.linalg.norm(e, dim=-1)
        x = r / rc
        inside = x < 1.0
        h = 1.0 + x ** 4 * (-35.0 + 84.0 * x - 70.0 * x ** 2 + 20.0 * x ** 3)
        dh = -140.0 * x ** 3 * (1.0 - x) ** 3 / rc
        k = n - 1 - l
        ez = norm * torch.exp(-zeta * r)
        f = ez * r ** k * h
        df = ez * ((k * r ** (k - 1) if k else 0.0) * h - zeta * r ** k * h + r ** k * dh)
        S, gS = _solid(l, m, e)
        u = torch.where(r > 1e-14, df * S / r.clamp_min(1e-14), torch.zeros_like(r))
        z = torch.zeros_like(r)
        out[0] += torch.where(inside, f * S, z)
        for i in range(3):
            out[1 + i] += torch.where(inside, u * e[..., i] + f * gS[i], z)
    return out


def _lag(t):
    """The four cubic Lagrange functions and their slopes at t, last axis."""
    nodes = [-1.0, -1.0 / 3.0, 1.0 / 3.0, 1.0]
    v, g = [], []
    for i in range(4):
        o = [nodes[j] for j in range(4) if j != i]
        c = 1.0 / ((nodes[i] - o[0]) * (nodes[i] - o[1]) * (nodes[i] - o[2]))
        a = [t - u for u in o]
        v.append(c * a[0] * a[1] * a[2])
        g.append(c * (a[0] * a[1] + a[0] * a[2] + a[1] * a[2]))
    return torch.stack(v, -1), torch.stack(g, -1)


def _fe_columns(xi, ser):
    """FE functions and reference gradients at xi (..., 3): (..., nfe), 3 x (..., nfe)."""
    if not ser:
        L, D = zip(*(_lag(xi[..., d]) for d in range(3)))
        prod = lambda x, y, z: (z[..., :, None, None] * y[..., None, :, None]
                                * x[..., None, None, :]).flatten(-3)
        return prod(*L), [prod(D[0], L[1], L[2]), prod(L[0], D[1], L[2]), prod(L[0], L[1], D[2])]
    at = [-1.0, -1.0 / 3.0, 1.0 / 3.0, 1.0]
    x = [xi[..., d] for d in range(3)]
    N, G = [], [[], [], []]
    for loc in range(64):
        i = (loc & 3, (loc >> 2) & 3, loc >> 4)
        inner = [d for d in range(3) if i[d] in (1, 2)]
        if len(inner) > 1:
            continue
        s = [at[j] for j in i]
        lin = [1.0 + s[d] * x[d] for d in range(3)]
        if not inner:
            q = 9.0 * (x[0] ** 2 + x[1] ** 2 + x[2] ** 2) - 19.0
            P = lin[0] * lin[1] * lin[2]
            N.append(P * q / 64.0)
            for d in range(3):
                o = lin[(d + 1) % 3] * lin[(d + 2) % 3]
                G[d].append((s[d] * o * q + 18.0 * P * x[d]) / 64.0)
            continue
        d = inner[0]
        a, b = (d + 1) % 3, (d + 2) % 3
        f = (1.0 - x[d] ** 2) * (1.0 + 9.0 * s[d] * x[d])
        fp = -2.0 * x[d] * (1.0 + 9.0 * s[d] * x[d]) + 9.0 * s[d] * (1.0 - x[d] ** 2)
        N.append(9.0 / 64.0 * f * lin[a] * lin[b])
        G[d].append(9.0 / 64.0 * fp * lin[a] * lin[b])
        G[a].append(9.0 / 64.0 * f * s[a] * lin[b])
        G[b].append(9.0 / 64.0 * f * lin[a] * s[b])
    return torch.stack(N, -1), [torch.stack(g, -1) for g in G]


class _Exact:
    """The elements in batches of equal column and point counts, each with its
    basis values, physical gradients, global columns and Bloch phases."""

    def __init__(self, s):
        self.s, self.wl, self.ctx = s, s["wl"], s["ctx"]
        self.dev = torch.device("cuda", torch.cuda.current_device())
        x, w, off = self.ctx.quadrature()
        self.x, self.w = torch.tensor(x, device=self.dev), torch.tensor(w, device=self.dev)
        n_e, dofs = self.ctx.element_basis()
        self.off, self.n_e = torch.tensor(off, device=self.dev), torch.tensor(n_e, device=self.dev).long()
        self.dofs = torch.tensor(dofs, device=self.dev).long()
        self.doff = torch.cumsum(self.n_e, 0) - self.n_e
        wl, nel = self.wl, int(self.wl["nel"])
        (self.L, self.inv), self.nel = _lattice_and_inverse(wl, self.dev), nel
        self.ser = wl.get("fe") == "serendipity32"
        # enrichment DOFs: by atom, orbital, vertex within r_e of the atom
        g = torch.arange(nel ** 3, device=self.dev)
        frac = torch.stack([g % nel, (g // nel) % nel, g // nel ** 2], 1).double() / nel
        kind, at, vert, self.types = [], [], [], []
        for ia, (sp, tau) in enumerate(wl["atoms"]):
            sp = wl["species"][sp]
            d = (frac @ self.L) - torch.tensor(tau, dtype=F64, device=self.dev)
            d = d - torch.round(d @ self.inv) @ self.L
            r = torch.linalg.norm(d[:, None, :] + _images(wl, 2 * sp["r_e"], self.dev), dim=2)
            v = torch.nonzero(r.min(dim=1).values <= sp["r_e"] + 1e-12)[:, 0]
            for o in sp["orbitals"]:
                key = (tuple(o), sp["r_c"])
                if key not in self.types:
                    self.types.append(key)
                kind.append(torch.full_like(v, self.types.index(key)))
                at.append(torch.full_like(v, ia))
                vert.append(v)
        self.n_fe = self.ctx.n_dof - sum(len(v) for v in vert)
        if self.n_fe != len(_node_positions(wl)):
            raise ValueError("the plan's enrichment columns are not those of the cell")
        cat = lambda v: torch.cat(v) if v else torch.zeros(0, dtype=torch.int64, device=self.dev)
        self.kind, self.at, self.vert = cat(kind), cat(at), cat(vert)
        self.tau = torch.tensor([t for _, t in wl["atoms"]], dtype=F64, device=self.dev).reshape(-1, 3)

    def batches(self, most=1 << 27):
        Q = self.off[1:] - self.off[:-1]
        key = self.n_e * (1 << 32) + Q
        for k in torch.unique(key).tolist():
            n, q = k >> 32, k & ((1 << 32) - 1)
            el = torch.nonzero(key == k)[:, 0]
            for c in torch.split(el, max(1, most // (5 * n * q))):
                yield self.batch(c, n, q)

    def batch(self, el, n, Q):
        nel, nfe = self.nel, 32 if self.ser else 64
        qi = self.off[el][:, None] + torch.arange(Q, device=self.dev)
        col = self.dofs[self.doff[el][:, None] + torch.arange(n, device=self.dev)]
        x, ec = self.x[qi], torch.stack([el % nel, (el // nel) % nel, el // nel ** 2], 1)
        Jinv = self.inv * 2.0 * nel     # d xi / d x
        xi = (x - (ec.double() / nel @ self.L)[:, None, :]) @ Jinv - 1.0
        B, G = _fe_columns(xi, self.ser)
        loc = torch.arange(64, device=self.dev)
        li = torch.stack([loc & 3, (loc >> 2) & 3, loc >> 4], 1)
        if self.ser:
            li = li[((li == 1) | (li == 2)).sum(1) <= 1]
        shift = (3 * ec[:, None, :] + li) // (3 * nel)
        if n > nfe:
            e = col[:, nfe:] - self.n_fe
            v = self.vert[e]
            vc = torch.stack([v % nel, (v // nel) % nel, v // nel ** 2], 2)
            up = vc != ec[:, None, :]                    # which of the two vertices per axis
            shift = torch.cat([shift, (ec[:, None, :] + up) // nel], 1)
            psi = torch.zeros(4, len(el), n - nfe, Q, dtype=F64, device=self.dev)
            for t, (orb, rc) in enumerate(self.types):
                i, j = torch.nonzero(self.kind[e] == t, as_tuple=True)
                for a in range(0, len(i), 1 << 15):
                    ii, jj = i[a:a + (1 << 15)], j[a:a + (1 << 15)]
                    d = x[ii] - self.tau[self.at[e[ii, jj]]][:, None, :]
                    psi[:, ii, jj] = torch.stack(_orbital(self.wl, orb, rc, d))
            psi = psi.transpose(2, 3)
            sg = (2.0 * up - 1.0).double()[:, None]      # E x 1 x cols x 3
            lin = 0.5 * (1.0 + sg * xi[:, :, None, :])
            phi = lin.prod(-1)
            dphi = [0.5 * sg[..., d] * lin[..., (d + 1) % 3] * lin[..., (d + 2) % 3] for d in range(3)]
            B = torch.cat([B, phi * psi[0]], 2)
            Gp = [sum(G[d] * Jinv[c, d] for d in range(3)) for c in range(3)]
            Gp = [torch.cat([Gp[c], sum(dphi[d] * Jinv[c, d] for d in range(3)) * psi[0]
                             + phi * psi[1 + c]], 2) for c in range(3)]
        else:
            Gp = [sum(G[d] * Jinv[c, d] for d in range(3)) for c in range(3)]
        ph = None
        if self.s["bloch"]:
            th = (shift.double() @ self.L) @ torch.tensor(self.s["k"], device=self.dev)
            ph = torch.polar(torch.ones_like(th), th)
        return qi, col, B, Gp, ph

    def everything(self, want):
        s, out = self.s, {}
        N = self.ctx.n_dof
        rowptr, pcol = self.ctx.pattern()
        rp = torch.tensor(rowptr, device=self.dev)
        row = torch.repeat_interleave(torch.arange(N, device=self.dev), rp[1:] - rp[:-1])
        keys = row * N + torch.tensor(pcol, device=self.dev)
        del row
        parts = 2 if s["bloch"] else 1
        zero = lambda n: [torch.zeros(n, dtype=F64, device=self.dev) for _ in range(parts)]
        V = s["V"].detach()
        H, S = zero(len(keys)), zero(len(keys)) if "S" in want else None
        rho = torch.zeros(self.ctx.n_q, dtype=F64, device=self.dev)
        vbar = torch.zeros_like(rho)
        for qi, col, B, G, ph in self.batches():
            w = self.w[qi][..., None]
            slot = torch.searchsorted(keys, col[:, :, None] * N + col[:, None, :])
            wB = w * B
            Se = B.transpose(1, 2) @ wB
            He = B.transpose(1, 2) @ (V[qi][..., None] * wB)
            for g in G:
                He += 0.5 * g.transpose(1, 2) @ (w * g)
            P = None if ph is None else ph.conj()[:, :, None] * ph[:, None, :]
            for M, to in ((He, H), (Se, S)):
                if to is None:
                    continue
                if P is None:
                    to[0].index_add_(0, slot.flatten(), M.flatten())
                else:
                    to[0].index_add_(0, slot.flatten(), (M * P.real).flatten())
                    to[1].index_add_(0, slot.flatten(), (M * P.imag).flatten())
            if "rho" in want:
                if ph is None:
                    psi2 = (B @ s["C"][col]) ** 2
                else:
                    c = torch.complex(s["C"][0][col], s["C"][1][col]) * ph[..., None]
                    psi2 = (B @ c.real) ** 2 + (B @ c.imag) ** 2
                rho[qi] = psi2 @ want["rho"]
            if "Vbar" in want:
                if ph is None:
                    Hb = s["Hbar"][slot]
                else:
                    Hb = s["Hbar"][0][slot] * P.real + s["Hbar"][1][slot] * P.imag
                vbar[qi] = ((B @ Hb) * wB).sum(-1)
        one = lambda v: v[0] if parts == 1 else tuple(v)
        out["H"] = one(H)
        if S is not None:
            out["S"] = one(S)
        out["rho"], out["Vbar"] = rho, vbar
        return out

    def project(self):
        s, wl = self.s, self.wl
        k = torch.tensor(s["k"], device=self.dev) if s["bloch"] else None
        val = torch.zeros(self.ctx.n_q, len(s["proj"]), dtype=torch.complex128, device=self.dev)
        for i, q in enumerate(s["proj"]):
            l, rp = q["l"], q["rp"]
            nrm = math.sqrt(2.0 / (math.gamma(l + 1.5) * rp ** (2 * l + 3)))
            d0 = self.x - torch.tensor(q["tau"], dtype=F64, device=self.dev)
            lat = torch.round(d0 @ self.inv) @ self.L
            for R in _images(wl, 9.6 * rp, self.dev):
                d = d0 - lat + R
                v = nrm * torch.exp(-(d * d).sum(1) / (2.0 * rp * rp)) * _solid(l, q["m"], d)[0]
                if k is None:
                    val[:, i] += v
                else:
                    val[:, i] += v * torch.polar(torch.ones_like(v), (lat - R) @ k)
        F = torch.zeros(self.ctx.n_dof, len(s["proj"]), dtype=torch.complex128, device=self.dev)
        for qi, col, B, _, ph in self.batches():
            t = (self.w[qi][..., None] * B).transpose(1, 2).to(torch.complex128) @ val[qi]
            if ph is not None:
                t = ph.conj()[..., None] * t
            F.index_add_(0, col.flatten(), t.flatten(0, 1))
        return dict(F=(F.real.contiguous(), F.imag.contiguous()) if s["bloch"] else F.real.contiguous())

    def coulomb(self, f):
        """V with -laplace V = 4 pi f, zero average, in the tricubic space."""
        nel, n = self.nel, 3 * self.nel
        h = float(self.wl["a"]) / nel
        t, wt = np.polynomial.legendre.leggauss(6)
        L, D = (v.numpy() for v in _lag(torch.tensor(t)))
        M, K = np.zeros((n, n)), np.zeros((n, n))
        for e in range(nel):
            i = (3 * e + np.arange(4)) % n
            np.add.at(M, (i[:, None], i), (L.T * wt) @ L * h / 2.0)
            np.add.at(K, (i[:, None], i), (D.T * wt) @ D * 2.0 / h)
        c = np.linalg.inv(np.linalg.cholesky(M))
        lam, X = np.linalg.eigh(c @ K @ c.T)
        X, lam = torch.tensor(c.T @ X, device=self.dev), torch.tensor(lam, device=self.dev)
        b = torch.zeros(n ** 3, dtype=F64, device=self.dev)
        for qi, col, B, _, _ in self.batches():
            b.index_add_(0, col[:, :64].flatten(),
                         (B[..., :64] * (self.w * f)[qi][..., None]).sum(1).flatten())
        b = 4.0 * math.pi * torch.einsum("zyx,zc,yb,xa->cba", b.view(n, n, n), X, X, X)
        den = lam[:, None, None] + lam[:, None] + lam
        den[0, 0, 0], b[0, 0, 0] = 1.0, 0.0
        v = torch.einsum("cba,zc,yb,xa->zyx", b / den, X, X, X).flatten()
        out = torch.empty_like(f)
        for qi, col, B, _, _ in self.batches():
            out[qi] = (B[..., :64] * v[col[:, None, :64]]).sum(-1)
        return out

    def scf(self):
        s, wl = self.s, self.wl
        eps, nelec = s["eps"], s["nelec"]
        occ = lambda mu: 2.0 / (1.0 + np.exp(np.clip((eps - mu) / KT, -700.0, 700.0)))
        lo, hi = eps.min() - 2.0, eps.max() + 2.0
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if occ(mid).sum() < nelec else (lo, mid)
        mu = 0.5 * (lo + hi)
        f = occ(mu)
        out = self.everything(dict(S=True, rho=torch.tensor(f, device=self.dev)))
        n_out, n_in, rho_I = out.pop("rho"), s["n_in"], s["rho_I"]
        out.pop("Vbar")

        def lda(n):
            rs = (3.0 / (4.0 * math.pi * n)) ** (1.0 / 3.0)
            ex = -0.75 * (3.0 * n / math.pi) ** (1.0 / 3.0)
            sq, lr = torch.sqrt(rs), torch.log(rs)
            e1 = -0.1423 / (1.0 + 1.0529 * sq + 0.3334 * rs)
            v1 = e1 * (1.0 + 7.0 / 6.0 * 1.0529 * sq + 4.0 / 3.0 * 0.3334 * rs) / (
                1.0 + 1.0529 * sq + 0.3334 * rs)
            e2 = 0.0311 * lr - 0.048 + 0.0020 * rs * lr - 0.0116 * rs
            v2 = (0.0311 * lr - 0.048 - 0.0311 / 3.0 + 2.0 / 3.0 * 0.0020 * rs * lr
                  + (-2.0 * 0.0116 - 0.0020) / 3.0 * rs)
            return (ex + torch.where(rs >= 1.0, e1, e2),
                    4.0 / 3.0 * ex + torch.where(rs >= 1.0, v1, v2))

        vc = self.coulomb(n_out - rho_I)
        w, V_in = self.w, s["V"]
        g = f / 2.0
        t = np.where((g > 1e-300) & (g < 1.0 - 1e-16),
                     g * np.log(np.maximum(g, 1e-300)) + (1.0 - g) * np.log1p(-np.minimum(g, 1 - 1e-16)), 0.0)
        info = dict(mu=mu, e_band=float((f * eps).sum()), e_dc=-float((w * n_out * V_in).sum()),
                    e_es=-0.5 * float((w * (rho_I - n_out) * vc).sum()),
                    e_self=sum(z * z / (sg * math.sqrt(2.0 * math.pi)) for z, sg in zip(*s["atoms"][1:])),
                    e_xc=float((w * n_out * lda(n_out)[0]).sum()), e_ts=2.0 * KT * float(t.sum()),
                    residual=float((w * (n_out - n_in).abs()).sum()))
        info["e_total"] = (info["e_band"] + info["e_dc"] + info["e_es"] - info["e_self"]
                           + info["e_xc"] + info["e_ts"])
        n = n_in + 0.5 * (n_out - n_in)
        out.update(n=n, V=self.coulomb(n - rho_I) + lda(n)[1], f=f, info=info)
        return out


def exact(case, seed):
    s = prepare(case, seed)
    x = _Exact(s)
    if s["call"] == "project":
        return x.project()
    if s["call"] == "scf":
        return x.scf()
    if s["call"] == "grad":
        out = x.everything(dict(Vbar=True))
        return dict(H=out["H"], V=out["Vbar"])
    want = dict(S=True, rho=s["f"])
    if s["call"] == "step":
        want["Vbar"] = True
    out = x.everything(want)
    return out if s["call"] == "step" else dict(H=out["H"], S=out["S"], rho=out["rho"])
