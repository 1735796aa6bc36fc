"""The first potential of a context on a stream that does not wait for the default
stream, while that one is busy: the load vector is cleared on the stream that solves.
The same values as on the default stream, to the order of the FP64 atomics (1e-12)."""
import numpy as np
import pytest

from paper_1611_00731_gb300 import pufe, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["c1_two_atom_4cube", "c2_rocksalt_6cube"])
def test_first_potential_on_a_stream_of_its_own(name):
    wl = W.workload(name)
    dev = torch.device("cuda:0")
    busy = torch.randn(4096, 4096, device=dev)
    got = []
    for own in (False, True):
        ctx = pufe.pufe_build_mesh(wl)
        rng = np.random.default_rng(121)
        n, rho = (torch.tensor(rng.uniform(0.2, 1.0, ctx.n_q), device=dev) for _ in range(2))
        V = torch.full((ctx.n_q,), float("nan"), dtype=torch.float64, device=dev)
        stream = torch.cuda.Stream() if own else torch.cuda.current_stream()
        torch.cuda.synchronize()
        for _ in range(20):   # the default stream has work for some milliseconds
            busy = busy @ busy
            busy /= busy.norm()
        ctx.pufe_effective_potential(n, rho, V, stream=stream)
        ctx.pufe_sync_status(stream=stream)
        torch.cuda.synchronize()
        got.append(V.cpu().numpy())
        ctx.close()
    assert np.isfinite(got[0]).all()
    assert np.abs(got[1] - got[0]).max() < 1e-12 * np.abs(got[0]).max()
