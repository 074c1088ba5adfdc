"""Ranges of the frequency grid's fixed-point histogram (mixed precision) against
the FP64 call, which bins alike: pole energies outside the bins, and weights whose sums are near
or past the ends of FP32; and widths of the histogram."""
import numpy as np
import pytest

from paper_2005_00827_gb300 import api, inputs
from tests.test_gpu_sigma_images import assert_every_patch, sigma

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("z", [2.4, 2.9, -2.9])
@pytest.mark.parametrize("sym", [True, False])
def test_weights_above_z_max(z, sym):
    """Quasi-particle lines with |Z| > z_max = 2 (24 is the last binned energy, 34.8
    the last pole): Sigma at |w| <= 3."""
    N, w = 8, np.linspace(-3.0, 3.0, 9)
    V, Z = inputs.random_vertex(N, 2.0, seed=1, c4v=sym), np.full(N, z)
    ref, got = (sigma(N, 4, 6, 0.0, 1, p, V, Z, 0.2, w) for p in (api.QPFRG_FP64, api.QPFRG_MIXED))
    assert_every_patch(got, ref)


@pytest.mark.parametrize("e", [-50, -45, -36, -33, -30, 30, 50])
def test_scaled_vertex(e):
    """Sigma is quadratic in V: the histogram's scale follows the vertex, also where
    the sum of a block's weights is near the end of FP32's range."""
    N, w = 12, np.linspace(-3.0, 3.0, 9)
    V, Z = inputs.random_vertex(N, 2.0, seed=4, c4v=False), inputs.z_profile(N, "aniso")
    ref, got = (sigma(N, 5, 4, 0.0, 0, api.QPFRG_MIXED, V * s, Z, 0.2, w) for s in (1.0, 2.0 ** e))
    assert_every_patch(got * 2.0 ** (-2 * e), ref)


@pytest.mark.parametrize("big", [3e19, -3e19, 1e30])
def test_overflowing_weight_is_not_finite(big):
    """A finite entry whose square leaves FP32: its target has no finite value, the
    others theirs."""
    N, w = 8, np.linspace(-3.0, 3.0, 9)
    V, Z = inputs.random_vertex(N, 2.0, seed=4, c4v=False), np.ones(N)
    ref = sigma(N, 4, 4, 0.0, 0, api.QPFRG_MIXED, V, Z, 0.2, w)
    V[5, 2, 3] = big
    got = sigma(N, 4, 4, 0.0, 0, api.QPFRG_MIXED, V, Z, 0.2, w)
    rest = np.arange(N) != 5
    assert not np.isfinite(got[5]).any()
    assert_every_patch(got[rest], ref[rest])


def test_overflowing_symmetric_vertex_is_not_finite():
    N, w = 8, np.linspace(-3.0, 3.0, 9)
    got = sigma(N, 4, 4, 0.0, 0, api.QPFRG_MIXED, np.full((N, N, N), 2e19), np.ones(N), 0.2, w)
    assert not np.isfinite(got).any()


def grid_ms(eta, V, Z, nt, nr, n=5):
    import torch
    N = len(Z)
    re, im = (torch.zeros(N, 9, dtype=torch.float64, device="cuda") for _ in range(2))
    V, Z, ms = torch.from_numpy(V.ravel()).cuda(), torch.from_numpy(Z).cuda(), []
    with api.Context(N, nt, nr, U=2.0, precision=api.QPFRG_MIXED, eta=eta, n_omega=9, omega_min=-3.0, omega_max=3.0) as c:
        for _ in range(n):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            api.qpfrg_selfenergy(c.h, 0.2, V, Z, re, im, None)
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
    return min(ms)


# bins: 96 / eta at t' = 0
@pytest.mark.parametrize("eta", [0.01614, 0.01612, 0.0135, 0.0134, 0.011, 0.00807, 0.0080])
def test_widths_of_the_histogram(eta):
    """Every number of words around the limits of one and of two histograms a CTA; a
    pole's FP32 energy is off by 2e-6 at most, of eta."""
    N, w = 8, np.linspace(-3.0, 3.0, 9)
    V, Z = inputs.random_vertex(N, 2.0, seed=4, c4v=False), inputs.z_profile(N, "aniso")
    ref, got = (sigma(N, 4, 6, 0.0, 0, p, V, Z, 0.2, w, eta) for p in (api.QPFRG_FP64, api.QPFRG_MIXED))
    assert (np.abs(got - ref).max(axis=1) < 2e-6 / eta * np.abs(ref).max(axis=1)).all()


@pytest.mark.parametrize("eta", [0.0138, 0.0131, 0.0128])
def test_no_cliff_in_eta(eta):
    """The table kernel serves these widths: two walks of the pairs and the flushes."""
    V, Z = inputs.random_vertex(24, 2.0, seed=4), inputs.z_profile(24, "aniso")
    assert grid_ms(eta, V, Z, 8, 8) < 4 * grid_ms(0.0165, V, Z, 8, 8)
