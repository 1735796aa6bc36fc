"""FP64 adjoint of elements with many enrichment columns in slots of one vertex each,
the direct form of the enrichment block, against the FP64 oracle: 163 and 164 columns
(the last block that goes through shared memory whole and the first that is cut into
ranges of rows), 186 (a whole block is beyond an SM's shared memory), 240, 448 (fewer
points at a time) and 907 and 908 (the last in ranges, the first in the pair form).  Tolerance 1e-12 of the largest
entry, as in the other FP64 parity tests."""
import itertools
import math

import numpy as np
import pytest
import scipy.sparse as sp

from oracle import assemble as oasm, bloch as ob, mesh as omesh, quadrature as oq
from paper_1611_00731_gb300 import pufe, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def one_vertex_slots(total):
    """2^3 elements, an atom on each of the 8 vertices that enriches only its own one:
    `total` slots of one vertex column on every element, 4^3 points."""
    shells = [(n, l, m, 1.0 + 0.25 * n + 0.125 * l) for n in range(1, 9) for l in range(min(n, 4))
              for m in range(-l, l + 1)]
    orbitals = shells + [(n, l, m, z + 0.0625) for n, l, m, z in shells]
    count = [total // 8 + (i < total % 8) for i in range(8)]
    return dict(name=f"one_vertex_slots_{total}", a=4.0, nel=2,
                species=[dict(name="X", Z=1.0, sigma=0.5, orbitals=orbitals[:c], r_c=1.9, r_e=0.5)
                         for c in count],
                atoms=[(i, tuple(2.0 * c for c in v))
                       for i, v in enumerate(itertools.product(range(2), repeat=3))],
                quad=dict(mode=W.QUAD_FIXED, p_far=4, p_near=4, p_min=0, p_max=0, tol=1e-6,
                          max_depth=0),
                nocc=2, nelec=4.0)


@pytest.mark.parametrize("total,bloch", [(163, True), (164, True), (186, False), (240, True),
                                         (448, False), (907, False), (908, False)])
def test_adjoint_of_many_one_vertex_slots(total, bloch):
    wl = one_vertex_slots(total)
    m = omesh.Mesh(wl)
    rules = oq.all_rules(m)
    ctx = pufe.pufe_build_mesh(wl)
    n_e, _ = ctx.element_basis()
    assert n_e.min() == n_e.max() == 64 + total
    assert set(ctx.element_slots().tolist()) == {total}
    ctx.pufe_tabulate(pufe.PUFE_FP64)
    rowptr, col = ctx.pattern()
    csr = lambda v: sp.csr_matrix((v, col, rowptr), shape=(ctx.n_dof, ctx.n_dof))
    up = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda:0")
    hr, hi = (W.random_symmetric_values(ctx.nnz, seed=s) for s in (61, 62))
    out = torch.full((ctx.n_q,), float("nan"), dtype=torch.float64, device="cuda:0")
    if bloch:
        k = 2.0 * math.pi / wl["a"] * np.array([0.3, -0.2, 0.1])
        ctx.pufe_assemble_HV_adjoint_bloch(k, up(hr), up(hi), out)
        ref = ob.adjoint_V_k(m, rules, csr(hr + 1j * hi), k)
    else:
        ctx.pufe_assemble_HV_adjoint(up(hr), out)
        ref = oasm.adjoint_V(m, rules, csr(hr))
    ctx.pufe_sync_status()
    assert float(np.abs(out.cpu().numpy() - ref).max() / np.abs(ref).max()) < 1e-12
