"""Row orbits under C4v and exchange with pairs that break the covariance of the
partner maps (momenta on a boundary between patches or shells, decided by
rounding): such pairs are rows for themselves, and the expanded right-hand side is
that of the unreduced launch in every precision."""
import numpy as np
import pytest

from paper_2005_00827_gb300 import api, inputs

pytestmark = pytest.mark.gpu

# the reduced and the unreduced launch sum the same loop kernels in other orders:
# rounding of FP64 sums of 1e4 terms, FP32 fixed-point rows and BF16 pairs
TOL = {api.QPFRG_FP64: 1e-12, api.QPFRG_MIXED: 5e-6, api.QPFRG_MIXED_TC: 2e-5}


@pytest.mark.parametrize("prec", list(TOL))
@pytest.mark.parametrize("N,nt,nr,ns,tp,reg", [
    (8, 2, 4, 1, 0.0, 0), (12, 3, 2, 1, 0.0, 0), (20, 4, 6, 1, -0.1, 0), (36, 5, 4, 1, 0.0, 0), (60, 10, 4, 1, -0.1, 0),
    (24, 2, 2, 3, 0.0, 0), (60, 4, 4, 5, 0.0, 0), (56, 2, 2, 7, 0.0, 1), (64, 2, 4, 1, 0.0, 1)])
def test_row_orbits_match_every_row(N, nt, nr, ns, tp, reg, prec):
    import torch
    lam = 0.3 if reg == 0 else 0.7
    V = inputs.random_vertex(N, 2.0, seed=N, n_shell=ns)
    Z = inputs.z_profile(N, "aniso", n_shell=ns)
    out, work = {}, {}
    for nosym in (0, 1):
        with api.Context(N, nt, nr, U=2.0, lambda0=lam, tp=tp, n_shell=ns, regulator=reg, T_fixed=0.2, precision=prec,
                         mode=api.QPFRG_GRID_SHELL if ns > 1 else api.QPFRG_GRID_WEDGE, no_loop_symmetry=nosym,
                         **(dict(step=0.01, lambda_end=2.0) if reg else {})) as c:
            dV = torch.full((N ** 3,), float("nan"), dtype=torch.float64, device="cuda")
            api.qpfrg_rhs(c.h, lam, torch.from_numpy(V.ravel()).cuda(), torch.from_numpy(Z).cuda(), dV)
            torch.cuda.synchronize()
            out[nosym], work[nosym] = dV.cpu().numpy(), api.qpfrg_rhs_work(c.h)
    assert np.abs(out[0] - out[1]).max() < TOL[prec] * np.abs(out[1]).max()
    assert work[0]["contraction_rows"] <= N * N and work[1]["contraction_rows"] == N * N
