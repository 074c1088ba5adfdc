"""FP64 and FP32 (SIMT) contraction against the FP64 oracle at the edges of its
tiles: 16 TM x 16 NB rows and columns, 16-wide blocks of the reduction, the
split over loop patches, odd lattices, single channels, and the forms chosen on
the device (representative rows for a C4v-symmetric input, every row for any
other, including an input that is symmetric but for one entry or one weight).
"""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2005_00827_gb300 import api, inputs

pytestmark = pytest.mark.gpu

# FP64: the sums have at most 2 N^2 <= 9 000 terms of relative rounding 1.1e-16,
# growing at most with their number: 1e-12.  FP32: loop kernels of 1e-6 and the
# same count of terms at 6e-8, growing with its root: 1e-5.
TOL = {api.QPFRG_FP64: 1e-12, api.QPFRG_MIXED: 1e-5}
W, L, S = api.QPFRG_GRID_WEDGE, api.QPFRG_GRID_LATTICE, api.QPFRG_GRID_SHELL


def rhs(ctx, T, V, Z):
    import torch
    dV = torch.full((V.size,), float("nan"), dtype=torch.float64, device="cuda")
    api.qpfrg_rhs(ctx.h, T, torch.from_numpy(V.ravel().copy()).cuda(), torch.from_numpy(Z.copy()).cuda(), dV)
    torch.cuda.synchronize()
    return dV.cpu().numpy().reshape(V.shape)


def off(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("prec", [api.QPFRG_FP64, api.QPFRG_MIXED])
@pytest.mark.parametrize("N,nt,nr,mode,ns,ch", [
    (4, 2, 2, W, 1, 7), (12, 2, 4, W, 1, 7), (20, 3, 2, W, 1, 7), (32, 2, 2, W, 1, 7), (36, 2, 2, W, 1, 7),
    (52, 2, 2, W, 1, 7), (9, 1, 1, L, 1, 7), (25, 1, 1, L, 1, 7), (1, 1, 1, L, 1, 7), (60, 2, 2, S, 5, 7),
    (16, 4, 4, W, 1, 1), (16, 4, 4, W, 1, 2), (16, 4, 4, W, 1, 4), (16, 4, 4, W, 1, 5), (16, 4, 4, W, 1, 0)])
@pytest.mark.parametrize("kind", ["sym", "asym", "one_entry", "one_weight"])
def test_contraction_edges(N, nt, nr, mode, ns, ch, prec, kind):
    T = 0.3
    rng = np.random.default_rng(N + ch)
    sym = kind != "asym" and mode != L
    V = inputs.random_vertex(N, 2.0, seed=N, c4v=sym, n_shell=ns) if mode != L else 2.0 + rng.random((N, N, N))
    Z = inputs.z_profile(N, "aniso", n_shell=ns) if sym else 0.8 + 0.2 * rng.random(N)
    if kind == "one_entry":
        V[N // 3, N // 2, N - 1] *= 1.01
    if kind == "one_weight":
        Z[N // 2] *= 1.01
    ref = Oracle(N, nt, nr, mode=mode, channels=ch, n_shell=ns).rhs(T, V, Z)
    with api.Context(N, nt, nr, U=2.0, mode=mode, precision=prec, channel_mask=ch, n_shell=ns) as ctx:
        got = rhs(ctx, T, V, Z)
        rows = api.qpfrg_rhs_work(ctx.h)
    if ch == 0:
        assert np.all(got == 0.0)
        return
    assert off(got, ref) < TOL[prec]
    if mode == W and nt % 2 == 0:
        assert (rows["contraction_rows"] < N * N) == (kind == "sym")


@pytest.mark.parametrize("prec", [api.QPFRG_FP64, api.QPFRG_MIXED])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_vertex_takes_every_row(prec, bad):
    """A NaN or infinity in a symmetric vertex spreads as in the sums themselves."""
    N, T = 16, 0.3
    V = inputs.random_vertex(N, 2.0, seed=3)
    V[1, 2, 3] = bad
    Z = inputs.z_profile(N, "aniso")
    with api.Context(N, 4, 4, U=2.0, precision=prec) as a, api.Context(N, 4, 4, U=2.0, precision=prec, no_loop_symmetry=1) as b:
        assert np.array_equal(np.isfinite(rhs(a, T, V, Z)), np.isfinite(rhs(b, T, V, Z)))


@pytest.mark.parametrize("prec", [api.QPFRG_FP64, api.QPFRG_MIXED])
def test_rhs_in_a_graph_follows_its_inputs(prec):
    """The form is decided on the device: a captured right-hand side replayed on
    other inputs in the same buffers gives theirs."""
    import torch
    N, T = 16, 0.3
    sym, asym = (inputs.random_vertex(N, 2.0, seed=5, c4v=c) for c in (True, False))
    Z = torch.from_numpy(inputs.z_profile(N, "aniso")).cuda()
    V = torch.from_numpy(sym.ravel().copy()).cuda()
    dV = torch.zeros_like(V)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with api.Context(N, 4, 4, U=2.0, precision=prec, stream=s.cuda_stream) as ctx:
        api.qpfrg_rhs(ctx.h, T, V, Z, dV)        # plans
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            api.qpfrg_rhs(ctx.h, T, V, Z, dV)
        for v in (asym, sym):
            V.copy_(torch.from_numpy(v.ravel().copy()))
            g.replay()
            torch.cuda.synchronize()
            got = dV.cpu().numpy().reshape(N, N, N)
            ref = Oracle(N, 4, 4).rhs(T, v, Z.cpu().numpy())
            assert off(got, ref) < TOL[prec]
