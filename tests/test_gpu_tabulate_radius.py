"""Rounding of the radius in the FP64 tabulation, seen through the exponential of a
sharp orbital (zeta = 128: the last place of a radius between 1 and 2 is 256 u of the
orbital, u = 2^-53).

Every number on the way to the radius is exact: the points are the centres of the
elements (one per axis) of a cell with dyadic edges, the atom's position and zeta are
dyadic.  The vertices' factors of 1/8 add up to 1 exactly, so the density of the state
with coefficient 1 on every vertex is the square of the orbital.  The reference takes
the correctly rounded root and everything after it in extended precision, so what is
left are the exponential (2 u), the cutoff at up to a quarter of its radius (3 u), the
norm (3 u), the harmonic's constant (u) and three products (3 u): 12 u, allowed 16 u;
the square doubles that and rounds once more."""
import numpy as np
import pytest

from paper_1611_00731_gb300 import pufe, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [(0.0, 0.0, 0.0), (3 / 64, 11 / 64, 29 / 64), (5 / 128, 1 / 32, 0.0)])
def test_radius_is_the_rounded_root(tau):
    zeta, rc, re = 128.0, 8.0, 2.5
    wl = dict(name="sharp_1s", a=8.0, nel=16,
              species=[dict(name="X", Z=1.0, sigma=0.5, orbitals=[(1, 0, 0, zeta)], r_c=rc, r_e=re)],
              atoms=[(0, tau)],
              quad=dict(mode=W.QUAD_FIXED, p_far=1, p_near=1, p_min=0, p_max=0, tol=1e-6,
                        max_depth=0),
              nocc=1, nelec=2.0)
    ctx = pufe.pufe_build_mesh(wl)
    x, _, _ = ctx.quadrature()
    assert np.array_equal(x, np.round(x * 4) / 4)
    ctx.pufe_tabulate(pufe.PUFE_FP64)
    C = np.zeros((ctx.n_dof, 1))
    C[48 ** 3:] = 1.0
    f, rho = torch.ones(1, dtype=torch.float64, device="cuda:0"), torch.empty(
        ctx.n_q, dtype=torch.float64, device="cuda:0")
    ctx.pufe_density(torch.tensor(C, device="cuda:0"), f, rho)
    ctx.pufe_sync_status()
    d = x - np.array(tau)
    d -= 8.0 * np.round(d / 8.0)
    r2 = (d ** 2).sum(axis=1)
    assert np.array_equal(r2, (d.astype(np.longdouble) ** 2).sum(axis=1))
    near = r2 <= 4
    r = np.sqrt(r2[near]).astype(np.longdouble)
    t = r / rc
    psi = (np.longdouble(2 * zeta) ** np.longdouble(1.5) / np.sqrt(np.longdouble(2)) * np.exp(-zeta * r)
           / np.sqrt(4 * np.longdouble("3.14159265358979323846264338327950288"))
           * (1 + t ** 4 * (-35 + t * (84 + t * (-70 + 20 * t)))))
    err = np.abs(rho.cpu().numpy()[near] / (psi * psi) - 1).astype(np.float64) / 2.0 ** -53
    assert near.sum() > 200 and err.max() <= 2 * 16 + 1, (near.sum(), err.max())
