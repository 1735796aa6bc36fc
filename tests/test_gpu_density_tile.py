"""The FP32 density of 64 to 128 real columns (its tiled product, `k_density_tile_f32`)
where it can go wrong: 32 to 64 complex states, so that the padding to groups of 8
states is empty, partly filled or all but empty and the groups are 8, 10, 12, 14 or 16
to a CTA; rows of C longer than the states that the call takes; 57 to 64 real states;
elements with and without more than 128 functions.  Against the FP64 oracle at 1e-5 of
the largest value, the mixed density's bound elsewhere."""
import ctypes
import math

import numpy as np
import pytest

from oracle import assemble as oasm, bloch as ob, mesh as omesh, quadrature as oq
from paper_1611_00731_gb300 import pufe, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _large_elements():
    """CsCl-like 4^3 cell with Ce-like orbitals of n >= 3: elements above 128 functions."""
    wl = W.workload("c3_cscl_4cube")
    wl["species"][0]["orbitals"] = [o for o in wl["species"][0]["orbitals"] if o[0] >= 3]
    wl["species"][0]["r_e"] = 1.5
    wl["quad"] = dict(wl["quad"], mode=W.QUAD_FIXED, p_far=5, p_near=5)
    return wl


CELLS = {"two_atom": lambda: dict(W.workload("c1_two_atom_4cube"), nel=5),
         "large_elements": _large_elements}


@pytest.fixture(scope="module", params=list(CELLS))
def cell(request):
    wl = CELLS[request.param]()
    m = omesh.Mesh(wl)
    ctx = pufe.pufe_build_mesh(wl)
    assert (ctx.max_basis > 128) == (request.param == "large_elements")
    ctx.pufe_tabulate(pufe.PUFE_TF32X3)
    return wl, m, oq.all_rules(m), ctx


def _call(fn, *args):
    status = fn(*(a.data_ptr() if torch.is_tensor(a) else a for a in args))
    assert status == 0, pufe.load_library().pufe_last_error().decode()


def _off(rho, ref):
    return float(np.abs(rho.cpu().numpy() - ref).max() / np.abs(ref).max())


@pytest.mark.parametrize("nocc", [32, 33, 41, 48, 49, 57, 63, 64])
def test_complex_states(cell, nocc):
    wl, m, rules, ctx = cell
    lib, ld = pufe.load_library(), nocc + 3
    k = 2.0 * math.pi / wl["a"] * np.array([0.3, -0.2, 0.1])
    kc = (ctypes.c_double * 3)(*k)
    Cr, Ci = (W.random_coefficients(ctx.n_dof, ld, seed=s) for s in (101, 102))
    f = W.random_occupations(nocc, seed=103)
    rho = torch.full((ctx.n_q,), float("nan"), dtype=torch.float64, device="cuda:0")
    _call(lib.pufe_density_bloch, ctx._h, kc, torch.tensor(Cr, device="cuda:0"),
          torch.tensor(Ci, device="cuda:0"), ld, torch.tensor(f, device="cuda:0"), nocc,
          pufe.PUFE_TF32X3, rho, torch.cuda.current_stream().cuda_stream)
    ctx.pufe_sync_status()
    assert _off(rho, ob.density_k(m, rules, (Cr + 1j * Ci)[:, :nocc], f, k)) < 1e-5


@pytest.mark.parametrize("nocc", [57, 64])
def test_real_states(cell, nocc):
    wl, m, rules, ctx = cell
    lib, ld = pufe.load_library(), nocc + 5
    C, f = W.random_coefficients(ctx.n_dof, ld, seed=104), W.random_occupations(nocc, seed=105)
    rho = torch.full((ctx.n_q,), float("nan"), dtype=torch.float64, device="cuda:0")
    _call(lib.pufe_density, ctx._h, torch.tensor(C, device="cuda:0"), ld,
          torch.tensor(f, device="cuda:0"), nocc, pufe.PUFE_TF32X3, rho,
          torch.cuda.current_stream().cuda_stream)
    ctx.pufe_sync_status()
    assert _off(rho, oasm.density(m, rules, C[:, :nocc], f)) < 1e-5
