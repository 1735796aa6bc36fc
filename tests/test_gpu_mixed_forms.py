"""FP32 FE-FE kernels, adjoint strip and tabulation of the mixed path at the sizes where
they can go wrong, against the FP64 oracle: the smallest and largest points per axis
(4 and 16), orders whose lines and rows do not fill the threads (5, 7, 11), one
element (every node repeated by periodicity), several images of an atom within its
cutoff and subdivided elements.  The mixed path's bounds: 5e-6 of the largest entry of
H and S, 1e-4 of the largest derivative."""
import math

import numpy as np
import pytest
import scipy.sparse as sp

from oracle import assemble as oasm, bloch as ob, mesh as omesh, quadrature as oq
from paper_1611_00731_gb300 import pufe, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HADAPT = dict(mode=W.QUAD_HADAPT, p_far=4, p_near=4, p_min=0, p_max=0, tol=1e-4, max_depth=2)

CELLS = {
    "p4": lambda: W.small_two_atom(nel=2, quad_p=4),
    "p5": lambda: W.small_two_atom(nel=2, quad_p=5),
    "p7_wide_support": lambda: W.small_two_atom(nel=2, quad_p=7, r_c=1.9, r_e=1.9),
    "p11": lambda: W.small_two_atom(nel=2, quad_p=11),
    "p16_one_element": lambda: W.small_two_atom(nel=1, quad_p=16),
    "images": lambda: W.small_two_atom(nel=2, a=2.0, quad_p=4, r_c=1.9, r_e=1.0),
    "subdivided": lambda: dict(W.small_two_atom(nel=2), quad=HADAPT),
}


@pytest.mark.parametrize("bloch", [False, True])
@pytest.mark.parametrize("name", list(CELLS))
def test_mixed_forms(name, bloch):
    wl = CELLS[name]()
    m = omesh.Mesh(wl)
    rules = oq.all_rules(m)
    ctx = pufe.pufe_build_mesh(wl)
    dev = torch.device("cuda:0")
    up = lambda a: torch.tensor(np.ascontiguousarray(a), device=dev)
    new = lambda n: torch.full((n,), float("nan"), dtype=torch.float64, device=dev)
    ctx.pufe_tabulate(pufe.PUFE_TF32X3)
    V = W.random_potential(ctx.n_q, seed=51)
    rowptr, col = ctx.pattern()
    csr = lambda v: sp.csr_matrix((v.cpu().numpy(), col, rowptr), shape=(ctx.n_dof, ctx.n_dof))
    off = lambda a, b: float(abs(a - b).max() / abs(b).max())
    rng = np.random.default_rng(52)
    vbar = new(ctx.n_q)
    if bloch:
        k = 2.0 * math.pi / wl["a"] * np.array([0.25, -0.125, 0.5])
        (Hr, Hi), (Sr, Si) = (new(ctx.nnz), new(ctx.nnz)), (new(ctx.nnz), new(ctx.nnz))
        ctx.pufe_assemble_HS_bloch(k, up(V), (Hr, Hi), (Sr, Si), prec=pufe.PUFE_TF32X3)
        H, S = csr(Hr) + 1j * csr(Hi), csr(Sr) + 1j * csr(Si)
        Ho, So = ob.assemble_HS_k(m, rules, V, k)
        Hbar = Ho.copy()
        Hbar.data = rng.standard_normal(Ho.nnz) + 1j * rng.standard_normal(Ho.nnz)
        ctx.pufe_assemble_HV_adjoint_bloch(k, up(Hbar.data.real), up(Hbar.data.imag), vbar,
                                           prec=pufe.PUFE_TF32X3)
        ref = ob.adjoint_V_k(m, rules, Hbar, k)
    else:
        h, s = new(ctx.nnz), new(ctx.nnz)
        ctx.pufe_assemble_HS(up(V), h, s, prec=pufe.PUFE_TF32X3)
        H, S = csr(h), csr(s)
        Ho, So = oasm.assemble_HS(m, rules, V)
        Hbar = Ho.copy()
        Hbar.data = rng.standard_normal(Ho.nnz)
        ctx.pufe_assemble_HV_adjoint(up(Hbar.data), vbar, prec=pufe.PUFE_TF32X3)
        ref = oasm.adjoint_V(m, rules, Hbar)
    ctx.pufe_sync_status()
    assert off(H, Ho) < 5e-6 and off(S, So) < 5e-6, (off(H, Ho), off(S, So))
    assert off(vbar.cpu().numpy(), ref) < 1e-4, off(vbar.cpu().numpy(), ref)


@pytest.mark.parametrize("nocc", [1, 8, 9])
@pytest.mark.parametrize("name", ["in_order", "p16_one_element", "images"])
def test_mixed_density_of_few_states(name, nocc):
    """The density of at most 8 states (its own form) and of one more, on elements whose
    vertices wrap around the cell and on ones whose slots run through them in order;
    1e-5 of the largest value, the mixed density's bound elsewhere."""
    wl = CELLS[name]() if name in CELLS else W.small_two_atom(nel=3, quad_p=4, r_c=1.9, r_e=1.9)
    m = omesh.Mesh(wl)
    rules = oq.all_rules(m)
    ctx = pufe.pufe_build_mesh(wl)
    ctx.pufe_tabulate(pufe.PUFE_TF32X3)
    C, f = W.random_coefficients(ctx.n_dof, nocc, seed=53), W.random_occupations(nocc, seed=54)
    dev = torch.device("cuda:0")
    rho = torch.full((ctx.n_q,), float("nan"), dtype=torch.float64, device=dev)
    ctx.pufe_density(torch.tensor(C, device=dev), torch.tensor(f, device=dev), rho,
                     prec=pufe.PUFE_TF32X3)
    ctx.pufe_sync_status()
    ref = oasm.density(m, rules, C, f)
    assert float(np.abs(rho.cpu().numpy() - ref).max() / np.abs(ref).max()) < 1e-5
