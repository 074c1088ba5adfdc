"""Patch counts N = 4 mod 8 at half filling without t': the lattice's mirror is a
boundary between wedges and percents of all pairs lie on it, decided by the FP64
projection's rounding.  Mixed precision against the FP64 call, every patch, and the
cost of a pair against a patch count that is a multiple of 8."""
import numpy as np
import pytest

from paper_2005_00827_gb300 import api, inputs
from tests.test_gpu_sigma_images import assert_every_patch

pytestmark = pytest.mark.gpu

# FP32 sums of 1e7 and more pairs, errors of 1e-5 each, independent (|slope| < 0.3)
TOL_Z = 1e-6


def run(N, nt, nr, prec, V, Z, w, n=1):
    import torch
    new = lambda *s: torch.full(s, float("nan"), dtype=torch.float64, device="cuda")  # noqa: E731
    with api.Context(N, nt, nr, U=2.0, precision=prec, eta=0.05, n_omega=len(w), omega_min=w[0], omega_max=w[-1]) as c:
        z, re, im = new(N), new(N, len(w)), new(N, len(w))
        V, Z = torch.from_numpy(V.ravel().copy()).cuda(), torch.from_numpy(Z).cuda()
        api.qpfrg_selfenergy(c.h, 0.2, V, Z, re, im, z)
        ms = []
        for _ in range(n):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            api.qpfrg_selfenergy(c.h, 0.2, V, Z, None, None, z)
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        torch.cuda.synchronize()
    return z.cpu().numpy(), re.cpu().numpy() + 1j * im.cpu().numpy(), min(ms)


@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("N,nt,nr", [(12, 16, 16), (20, 16, 8), (52, 4, 4), (28, 5, 6), (4, 24, 24)])
def test_every_patch(N, nt, nr, sym):
    w = np.linspace(-3.0, 3.0, 9)
    V, Z = inputs.random_vertex(N, 2.0, seed=N, c4v=sym), inputs.z_profile(N, "aniso")
    (zr, ref, _), (z, got, _) = (run(N, nt, nr, p, V, Z, w) for p in (api.QPFRG_FP64, api.QPFRG_MIXED))
    assert np.abs(z - zr).max() < TOL_Z
    assert_every_patch(got, ref)


@pytest.mark.parametrize("sym", [True, False])
def test_ties_cost_little(sym):
    """52 patches against the 48 patches that sum every patch: time per pair."""
    per = []
    for N, s in ((52, sym), (48, False)):
        V, Z = inputs.random_vertex(N, 2.0, seed=N, c4v=s), inputs.z_profile(N, "aniso")
        per.append(run(N, 8, 8, api.QPFRG_MIXED, V, Z, np.zeros(1), 5)[2] / N ** 3)
    assert per[0] < 3.5 * per[1]


def test_reduced_targets_pay_on_the_largest_grid():
    """96 patches, 32 x 32 points: 16 of 96 targets, a million boundary pairs."""
    import torch
    N, ms = 96, {}
    with api.Context(N, 32, 32, U=2.0, precision=api.QPFRG_MIXED, sigma_table=-1, n_omega=9, omega_min=-3.0,
                     omega_max=3.0) as c:
        z, re, im = (torch.zeros(*s, dtype=torch.float64, device="cuda") for s in ((N,), (N, 9), (N, 9)))
        Z = torch.from_numpy(inputs.z_profile(N, "aniso")).cuda()
        for sym in (True, False):
            V = torch.from_numpy(inputs.random_vertex(N, 2.0, seed=N, c4v=sym).ravel()).cuda()
            for name, args in (("Z", (None, None, z)), ("grid", (re, im, None))):
                api.qpfrg_selfenergy(c.h, 0.2, V, Z, *args)
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                api.qpfrg_selfenergy(c.h, 0.2, V, Z, *args)
                b.record()
                torch.cuda.synchronize()
                ms[name, sym] = a.elapsed_time(b)
    assert all(ms[n, True] < 0.3 * ms[n, False] for n in ("Z", "grid"))
