"""FP64 sum-factorized forms at the sizes where they can go wrong, against the
FP64 oracle: the smallest and largest points per axis (4 and 16) that the
factorized assembly takes and the 3 that it leaves to the direct kernel, one
element (every node repeated by periodicity), slots of one vertex column (the
direct enrichment blocks) and of eight (the pair form).  Tolerance 1e-12 of the
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
    "wide_support": lambda: W.small_two_atom(nel=3, quad_p=5, r_c=1.9, r_e=1.9),
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
    k = 2.0 * math.pi / wl["a"] * np.array([0.3, -0.2, 0.1])
    V = W.random_potential(ctx.n_q, seed=6)
    Ho, So = ob.assemble_HS_k(m, rules, V, k)
    mk = lambda: torch.full((ctx.nnz,), 3.0, dtype=torch.float64, device="cuda:0")
    H, S = (mk(), mk()), (mk(), mk())
    ctx.pufe_assemble_HS_bloch(k, _dev(V), H, S)
    ctx.pufe_sync_status()
    c = lambda v: _csr(ctx, v[0].cpu().numpy() + 1j * v[1].cpu().numpy())
    assert _off(c(H), Ho) < TOL
    assert _off(c(S), So) < TOL
