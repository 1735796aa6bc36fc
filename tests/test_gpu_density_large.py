"""FP64 density of elements with many functions on rules of 16 points per axis, where a
group of 16 columns does not fit shared memory: 428 functions and more, up to 3,392
with the most states that the call takes there (8), at the Gamma point and at a
wavevector, against the FP64 oracle.  Tolerance 1e-12 of the largest value, as in the
other FP64 parity tests."""
import math

import numpy as np
import pytest

from oracle import assemble as oasm, bloch as ob, mesh as omesh, quadrature as oq
from paper_1611_00731_gb300 import pufe, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def one_element(slots):
    """One element of 16^3 points and one atom whose `slots` orbitals each enrich the
    one vertex, eight times the element's: 64 + 8 slots functions."""
    shells = [(n, l, m, 1.0 + 0.25 * n + 0.125 * l) for n in range(1, 9) for l in range(min(n, 4))
              for m in range(-l, l + 1)]
    orbitals = [(n, l, m, z + 0.0625 * i) for i in range(5) for n, l, m, z in shells][:slots]
    return dict(name=f"one_element_{slots}", a=4.0, nel=1,
                species=[dict(name="X", Z=1.0, sigma=0.5, orbitals=orbitals, r_c=1.9, r_e=0.5)],
                atoms=[(0, (0.0, 0.0, 0.0))],
                quad=dict(mode=W.QUAD_FIXED, p_far=16, p_near=16, p_min=0, p_max=0, tol=1e-6,
                          max_depth=0),
                nocc=2, nelec=4.0)


# (slots, states at the Gamma point, states at the wavevector)
@pytest.mark.parametrize("slots,nocc,nocc_k", [(45, 16, 16), (46, 16, 16), (56, 13, 24),
                                               (56, 32, 7), (200, 13, 8), (416, 8, None)])
def test_density_of_many_functions(slots, nocc, nocc_k):
    wl = one_element(slots)
    m = omesh.Mesh(wl)
    rules = oq.all_rules(m)
    ctx = pufe.pufe_build_mesh(wl)
    assert ctx.max_basis == 64 + 8 * slots
    ctx.pufe_tabulate(pufe.PUFE_FP64)
    up = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda:0")
    off = lambda a, b: float(np.abs(a - b).max() / np.abs(b).max())
    rho = torch.full((ctx.n_q,), float("nan"), dtype=torch.float64, device="cuda:0")
    C, f = W.random_coefficients(ctx.n_dof, nocc, seed=71), W.random_occupations(nocc, seed=72)
    ctx.pufe_density(up(C), up(f), rho)
    ctx.pufe_sync_status()
    assert off(rho.cpu().numpy(), oasm.density(m, rules, C, f)) < 1e-12
    if nocc_k is None:
        return
    k = 2.0 * math.pi / wl["a"] * np.array([0.3, -0.2, 0.1])
    Cr, Ci = (W.random_coefficients(ctx.n_dof, nocc_k, seed=s) for s in (73, 74))
    f = W.random_occupations(nocc_k, seed=75)
    ctx.pufe_density_bloch(k, up(Cr), up(Ci), up(f), rho)
    ctx.pufe_sync_status()
    assert off(rho.cpu().numpy(), ob.density_k(m, rules, Cr + 1j * Ci, f, k)) < 1e-12
