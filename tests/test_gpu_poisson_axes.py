"""The Poisson solve on meshes with different node counts per axis, with the axis
matrices staged in shared memory (up to 96 nodes on the longest axis) and read in
place (more), the long axis on x, y or z.  Reference: the FE system assembled here as Kronecker products of the
1D periodic cubic elements and solved directly; 1e-10 of the largest value, as in the
other SCF tests."""
import ctypes as C
import math

import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spla

from oracle.fe import gauss_1d
from oracle.scf import pz81
from paper_1611_00731_gb300 import pufe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10
P = 4   # points per axis


def _build(nel, a):
    """A cell without atoms, nel[d] elements on axis d."""
    lib = pufe.load_library()
    cell = pufe._Cell((C.c_double * 3)(*a), (C.c_int * 3)(*nel), 0, (C.c_double * 1)(),
                      (C.c_int * 1)(), None, pufe.PUFE_FE_LAGRANGE64)
    quad = pufe._Quad(0, P, P, 0, 0, 1e-6, 0, 0)
    h = C.c_void_p()
    pufe._check(lib.pufe_build_mesh(C.byref(cell), (pufe._Species * 1)(), 0, C.byref(quad),
                                    C.byref(h)))
    return pufe.Context(h, dict(nel=nel, a=a))


def _lagrange(t):
    """Values and slopes of the four cubic Lagrange functions, (len(t), 4) each."""
    x = np.array([-1.0, -1.0 / 3.0, 1.0 / 3.0, 1.0])
    V = np.empty((len(t), 4))
    D = np.empty((len(t), 4))
    for i in range(4):
        c = np.poly1d(np.poly(np.delete(x, i)) / np.prod(x[i] - np.delete(x, i)))
        V[:, i], D[:, i] = c(t), c.deriv()(t)
    return V, D


def _axis(nel, h):
    """1D mass and stiffness (3 nel nodes, periodic) and the values of the 1D functions
    at the P nel Gauss points, sparse."""
    t, w = gauss_1d(4)
    V, D = _lagrange(t)
    Me, Ke = (V.T * w) @ V * (h / 2.0), (D.T * w) @ D * (2.0 / h)
    n = 3 * nel
    M, K = sp.lil_matrix((n, n)), sp.lil_matrix((n, n))
    B = sp.lil_matrix((P * nel, n))
    Vp, _ = _lagrange(gauss_1d(P)[0])
    for e in range(nel):
        for i in range(4):
            gi = (3 * e + i) % n
            for q in range(P):
                B[P * e + q, gi] += Vp[q, i]
            for j in range(4):
                gj = (3 * e + j) % n
                M[gi, gj] += Me[i, j]
                K[gi, gj] += Ke[i, j]
    return M.tocsr(), K.tocsr(), B.tocsr()


def _reference(nel, a, w, f):
    """V_C at the points (element order) with del^2 V_C = -4 pi f and zero cell average."""
    ax = [_axis(n, L / n) for n, L in zip(nel, a)]
    kron = lambda x, y, z: sp.kron(sp.kron(z, y), x, format="csr")   # x fastest
    (Mx, Kx, Bx), (My, Ky, By), (Mz, Kz, Bz) = ax
    K = kron(Kx, My, Mz) + kron(Mx, Ky, Mz) + kron(Mx, My, Kz)
    B = kron(Bx, By, Bz)
    # element order (ex + nx (ey + ny ez), x fastest inside) -> grid order
    ne, g = nel[0] * nel[1] * nel[2], [P * n for n in nel]
    e, q = np.divmod(np.arange(ne * P ** 3), P ** 3)
    ix = P * (e % nel[0]) + q % P
    iy = P * ((e // nel[0]) % nel[1]) + (q // P) % P
    iz = P * (e // (nel[0] * nel[1])) + q // P ** 2
    at = ix + g[0] * (iy + g[1] * iz)
    load = np.zeros(len(at))
    load[at] = w * f
    ones = np.zeros(len(at))
    ones[at] = w
    b, m = B.T @ load, B.T @ ones
    b = 4.0 * math.pi * (b - b.sum() / m.sum() * m)
    Kp = K.tolil()
    Kp[0, :] = 0.0
    Kp[0, 0] = 1.0
    b[0] = 0.0
    v = spla.spsolve(Kp.tocsc(), b)
    v -= (m @ v) / m.sum()
    return (B @ v)[at]


def _case(nel):
    a = tuple(0.9 * n + 0.3 * d for d, n in enumerate(nel))
    ctx = _build(nel, a)
    _, w, _ = ctx.quadrature()
    rng = np.random.default_rng(111)
    n, rho = rng.uniform(0.1, 1.0, ctx.n_q), rng.uniform(0.1, 1.0, ctx.n_q)
    rho *= (w @ n) / (w @ rho)   # neutral
    return ctx, n, rho, _reference(nel, a, w, n - rho)


def _off(a, b):
    return float(np.abs(a.cpu().numpy() - b).max() / np.abs(b).max())


# 32 elements: 96 nodes, staged; 33: 99, read in place
@pytest.mark.parametrize("nel", [(2, 3, 4), (32, 2, 3), (3, 32, 1), (2, 1, 32), (33, 3, 2),
                                 (1, 33, 2), (2, 3, 33), (38, 2, 1), (1, 1, 1)])
def test_effective_potential_on_unequal_axes(nel):
    ctx, n, rho, ref = _case(nel)
    nd, rd = (torch.tensor(v, device="cuda:0") for v in (n, rho))
    V, VC, exc = (torch.full((ctx.n_q,), float("nan"), dtype=torch.float64, device="cuda:0")
                  for _ in range(3))
    for _ in range(2):   # (the second solve finds what the first one left)
        ctx.pufe_effective_potential(nd, rd, V, VC, exc)
        ctx.pufe_sync_status()
        e, v = pz81(n)
        assert _off(VC, ref) < TOL and _off(exc, e) < 1e-13 and _off(V, ref + v) < TOL
