"""What happens when a launch meets more pairs than it can note down: more guarded
pairs than the queue holds (every pair of the chunk is looked at again), more boundary
pairs than the record holds (every patch is summed).  The capacities are lowered by
the environment; results as with the full ones."""
import numpy as np
import pytest

from paper_2005_00827_gb300 import api, inputs
from tests.test_gpu_sigma_images import GEO

pytestmark = pytest.mark.gpu


def run(N, nt, nr, tp, prop, prec, V, Z, w):
    import torch
    new = lambda *s: torch.full(s, float("nan"), dtype=torch.float64, device="cuda")  # noqa: E731
    with api.Context(N, nt, nr, U=2.0, tp=tp, precision=prec, propagator=prop, eta=0.05, n_omega=len(w), omega_min=w[0],
                     omega_max=w[-1]) as c:
        z, re, im = new(N), new(N, len(w)), new(N, len(w))
        api.qpfrg_selfenergy(c.h, 0.2, torch.from_numpy(V.ravel().copy()).cuda(), torch.from_numpy(Z).cuda(), re, im, z)
        torch.cuda.synchronize()
    return z.cpu().numpy(), re.cpu().numpy() + 1j * im.cpu().numpy()


# sums in another order: FP32 rounding of partial sums (FP64 for the FP64 call)
REL = {api.QPFRG_FP64: 1e-12, api.QPFRG_MIXED: 2e-6}


@pytest.mark.parametrize("name,limit", [("QPFRG_TEST_QUEUE", 0), ("QPFRG_TEST_QUEUE", 7), ("QPFRG_TEST_BOUNDARY_PAIRS", 1)])
@pytest.mark.parametrize("prec", list(REL))
@pytest.mark.parametrize("geo", GEO + [(16, 20, 16, 0.0, 0), (8, 4, 4, -0.3, 0)], ids=lambda g: "_".join(map(str, g)))
def test_overrun_changes_nothing(geo, prec, name, limit, monkeypatch):
    N, nt, w = geo[0], geo[1], np.linspace(-3.0, 3.0, 9)
    V, Z = inputs.random_vertex(N, 2.0, seed=N + nt), inputs.z_profile(N, "aniso")
    z0, s0 = run(*geo, prec, V, Z, w)
    monkeypatch.setenv(name, str(limit))
    z1, s1 = run(*geo, prec, V, Z, w)
    assert np.abs(z1 - z0).max() < REL[prec]
    assert np.abs(s1 - s0).max() < REL[prec] * np.abs(s0).max()
