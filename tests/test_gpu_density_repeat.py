"""The FP64 density repeats bit for bit, whatever the number of columns (states at the
Gamma point, real and imaginary parts at a wavevector): one, two and more groups of up
to 16 columns, on elements whose (sub)cells are cut to fill the chip and on whole ones."""
import math

import numpy as np
import pytest

from paper_1611_00731_gb300 import pufe, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CELLS = {
    "eight_elements": lambda: W.small_two_atom(nel=2, quad_p=6),
    "p16_one_element": lambda: W.small_two_atom(nel=1, quad_p=16),
    "c1_two_atom_4cube": lambda: W.workload("c1_two_atom_4cube"),
}


@pytest.mark.parametrize("nocc", [8, 32, 33, 48, 64])
@pytest.mark.parametrize("name", list(CELLS))
def test_density_repeats(name, nocc):
    wl = CELLS[name]()
    ctx = pufe.pufe_build_mesh(wl)
    ctx.pufe_tabulate(pufe.PUFE_FP64)
    up = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda:0")
    Cr, Ci = (up(W.random_coefficients(ctx.n_dof, nocc, seed=s)) for s in (81, 82))
    f = up(W.random_occupations(nocc, seed=83))
    k = 2.0 * math.pi / wl["a"] * np.array([0.3, -0.2, 0.1])
    for call in (lambda out: ctx.pufe_density(Cr, f, out),
                 lambda out: ctx.pufe_density_bloch(k, Cr, Ci, f, out)):
        first = torch.full((ctx.n_q,), float("nan"), dtype=torch.float64, device="cuda:0")
        again = first.clone()
        call(first)
        for _ in range(20):
            call(again)
            assert torch.equal(first, again)
    ctx.pufe_sync_status()
