"""FP64 sum-factorized forms at the sizes where they can go wrong, against the
FP64 oracle: the smallest and largest points per axis (4 and 16) that the
factorized assembly takes and the 3 that it leaves to the direct kernel, one
element (every node repeated by periodicity), slots of one vertex column (the
direct enrichment blocks) and of eight (the pair form), several images of an atom
within its cutoff (the tabulation's sum), one state, an odd count
and the most that a call takes.  Tolerance 1e-12 of the
largest entry, as in the other FP64 parity tests."""
import math

import numpy as np
import pytest
import scipy.sparse as sp

from oracle import assemble as oasm, bloch as ob, mesh as omesh, quadrature as oq
from paper_1611_00731_gb300 import pufe, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-12

CELLS = {
    "p4": lambda: W.small_two_atom(nel=2, quad_p=4),
    "p3_direct_kernel": lambda: W.small_two_atom(nel=2, quad_p=3),
    "p9": lambda: W.small_two_atom(nel=2, quad_p=9),
    "p16_one_element": lambda: W.small_two_atom(nel=1, quad_p=16),
    "one_vertex_slots": lambda: W.small_two_atom(nel=3, quad_p=6, r_e=0.5),
    # (an even order: an odd one puts a point on the nucleus, where the oracle's
    # direction cosines are 0/0)
    # several periodic images within r_c of a point
    "images": lambda: W.small_two_atom(nel=2, a=2.0, quad_p=4, r_c=1.9, r_e=1.0),
    # general cells (the metric's cross terms) and the serendipity space (its rows
    # lifted to the tricubic ones), alone and together, in both E x E forms
    "triclinic": lambda: W.ceal_like(nel=2, quad_p=5),
    "triclinic_wide": lambda: W.ceal_like(nel=3, quad_p=4, r_c=3.0, r_e=2.9),
    "serendipity": lambda: dict(W.small_two_atom(nel=3, quad_p=6, r_c=1.9, r_e=1.9),
                                fe="serendipity32"),
    "triclinic_serendipity": lambda: dict(W.ceal_like(nel=2, quad_p=9), fe="serendipity32"),
    "serendipity_p3": lambda: dict(W.small_two_atom(nel=2, quad_p=3), fe="serendipity32"),
    "wide_support": lambda: W.small_two_atom(nel=3, quad_p=6, r_c=1.9, r_e=1.9),
}


@pytest.fixture(scope="module", params=list(CELLS))
def cell(request):
    wl = CELLS[request.param]()
    m = omesh.Mesh(wl)
    ctx = pufe.pufe_build_mesh(wl)
    ctx.pufe_tabulate(pufe.PUFE_FP64)
    return wl, m, oq.all_rules(m), ctx


def _dev(x):
    return torch.tensor(np.ascontiguousarray(x), device="cuda:0")


def _off(a, b):
    return float(abs(a - b).max() / abs(b).max())


def _csr(ctx, v):
    rowptr, col = ctx.pattern()
    return sp.csr_matrix((v, col, rowptr), shape=(ctx.n_dof, ctx.n_dof))


def test_assembly(cell):
    wl, m, rules, ctx = cell
    V = W.random_potential(ctx.n_q, seed=5)
    Ho, So = oasm.assemble_HS(m, rules, V)
    mk = lambda: torch.full((ctx.nnz,), 3.0, dtype=torch.float64, device="cuda:0")
    H, S, H1, S1 = mk(), mk(), mk(), mk()
    ctx.pufe_assemble_HS(_dev(V), H, S)
    ctx.pufe_assemble_HS(_dev(V), H1, None)
    ctx.pufe_assemble_HS(None, None, S1)
    ctx.pufe_sync_status()
    assert _off(_csr(ctx, H.cpu().numpy()), Ho) < TOL
    assert _off(_csr(ctx, S.cpu().numpy()), So) < TOL
    assert _off(_csr(ctx, H1.cpu().numpy()), Ho) < TOL
    assert _off(_csr(ctx, S1.cpu().numpy()), So) < TOL


def test_assembly_at_a_wavevector(cell):
    wl, m, rules, ctx = cell
    k = 2.0 * math.pi / (wl["a"] or W.CEAL_A) * np.array([0.3, -0.2, 0.1])
    V = W.random_potential(ctx.n_q, seed=6)
    Ho, So = ob.assemble_HS_k(m, rules, V, k)
    mk = lambda: torch.full((ctx.nnz,), 3.0, dtype=torch.float64, device="cuda:0")
    H, S = (mk(), mk()), (mk(), mk())
    ctx.pufe_assemble_HS_bloch(k, _dev(V), H, S)
    ctx.pufe_sync_status()
    c = lambda v: _csr(ctx, v[0].cpu().numpy() + 1j * v[1].cpu().numpy())
    assert _off(c(H), Ho) < TOL
    assert _off(c(S), So) < TOL


@pytest.mark.parametrize("nocc", [1, 17, 64])
def test_density(cell, nocc):
    wl, m, rules, ctx = cell
    Cm = W.random_coefficients(ctx.n_dof, nocc, seed=nocc)
    f = W.random_occupations(nocc, seed=nocc)
    rho = torch.full((ctx.n_q,), 3.0, dtype=torch.float64, device="cuda:0")
    ctx.pufe_density(_dev(Cm), _dev(f), rho)
    ctx.pufe_sync_status()
    assert _off(rho.cpu().numpy(), oasm.density(m, rules, Cm, f)) < TOL


def test_adjoint(cell):
    wl, m, rules, ctx = cell
    h = W.random_symmetric_values(ctx.nnz, seed=3)   # (not symmetrised: a general cotangent)
    v = torch.full((ctx.n_q,), 3.0, dtype=torch.float64, device="cuda:0")
    ctx.pufe_assemble_HV_adjoint(_dev(h), v)
    ctx.pufe_sync_status()
    assert _off(v.cpu().numpy(), oasm.adjoint_V(m, rules, _csr(ctx, h))) < TOL


def test_density_and_adjoint_at_a_wavevector(cell):
    wl, m, rules, ctx = cell
    k = 2.0 * math.pi / (wl["a"] or W.CEAL_A) * np.array([0.3, -0.2, 0.1])
    Cr, Ci = (W.random_coefficients(ctx.n_dof, 7, seed=s) for s in (1, 2))
    f = W.random_occupations(7, seed=3)
    hr, hi = (W.random_symmetric_values(ctx.nnz, seed=s) for s in (4, 5))
    out = [torch.full((ctx.n_q,), 3.0, dtype=torch.float64, device="cuda:0") for _ in range(2)]
    ctx.pufe_density_bloch(k, _dev(Cr), _dev(Ci), _dev(f), out[0])
    ctx.pufe_assemble_HV_adjoint_bloch(k, _dev(hr), _dev(hi), out[1])
    ctx.pufe_sync_status()
    assert _off(out[0].cpu().numpy(), ob.density_k(m, rules, Cr + 1j * Ci, f, k)) < TOL
    assert _off(out[1].cpu().numpy(), ob.adjoint_V_k(m, rules, _csr(ctx, hr + 1j * hi), k)) < TOL
