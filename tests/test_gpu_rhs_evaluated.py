"""What a right-hand side computes (qpfrg_rhs_evaluated): on the row orbits one table
row per orbit of transfer pairs under C4v and exchange, counted once though two
contraction rows may share it; pairs that break covariance are rows of their own and
keep the form compact; other inputs every row."""
import numpy as np
import pytest

from paper_2005_00827_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def counts(N, nt, nr, prec, V, n_shell=1, tp=0.0):
    import torch
    with api.Context(N, nt, nr, U=2.0, tp=tp, precision=prec, n_shell=n_shell,
                     mode=api.QPFRG_GRID_SHELL if n_shell > 1 else api.QPFRG_GRID_WEDGE) as c:
        dV = torch.zeros(N ** 3, dtype=torch.float64, device="cuda")
        Z = torch.from_numpy(inputs.z_profile(N, "aniso", n_shell=n_shell)).cuda()
        api.qpfrg_rhs(c.h, 0.3, torch.from_numpy(V.ravel().copy()).cuda(), Z, dV)
        return api.qpfrg_rhs_evaluated(c.h), api.qpfrg_rhs_work(c.h)


@pytest.mark.parametrize("prec", [api.QPFRG_FP64, api.QPFRG_MIXED, api.QPFRG_MIXED_TC])
@pytest.mark.parametrize("N,nt,nr", [(8, 2, 4), (16, 4, 4), (32, 2, 2)])
def test_symmetric_vertex(N, nt, nr, prec):
    ev, work = counts(N, nt, nr, prec, inputs.random_vertex(N, 2.0, seed=N))
    maps = inputs.c4v_patch_maps(N)
    orbits = {min(min(g[x] * N + g[y], g[y] * N + g[x]) for g in maps) for x in range(N) for y in range(N)}
    assert ev == dict(loop_evals=2 * len(orbits) * N * nt * nr, table_rows=len(orbits))
    assert len(orbits) < work["contraction_rows"] < N * N and ev["loop_evals"] < work["loop_evals"]


@pytest.mark.parametrize("prec", [api.QPFRG_FP64, api.QPFRG_MIXED, api.QPFRG_MIXED_TC])
@pytest.mark.parametrize("N,nt,nr,ns,tp", [(12, 3, 2, 1, 0.0), (20, 4, 6, 1, -0.1), (36, 5, 4, 1, 0.0), (60, 10, 4, 1, -0.1),
                                           (24, 2, 2, 3, 0.0), (60, 4, 4, 5, 0.0), (56, 2, 2, 7, 0.0)])
def test_pairs_that_break_covariance_stay_compact(N, nt, nr, ns, tp, prec):
    """The geometries whose right-hand sides are compared with every row (row orbits)."""
    ev, work = counts(N, nt, nr, prec, inputs.random_vertex(N, 2.0, seed=N, n_shell=ns), ns, tp)
    assert work["rows_unreduced"] > 0
    assert ev["table_rows"] < work["contraction_rows"] < N * N / 2


def test_unsymmetric_vertex():
    N = 16
    ev, work = counts(N, 4, 4, api.QPFRG_MIXED, inputs.random_vertex(N, 2.0, seed=N, c4v=False))
    assert work["contraction_rows"] == ev["table_rows"] == N * N and ev["loop_evals"] == work["loop_evals"]
