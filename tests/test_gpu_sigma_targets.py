"""FP32 self-energies of the wedge grid with their targets chosen on the device
(irreducible and zone-edge patches of a C4v-symmetric vertex, every patch of any
other), the fixed-point frequency histogram and the interaction flow's line
weights, against the FP64 oracle: odd and ragged grids, passes of more than 256 records,
loop-point counts that leave a partial block, t' != 0, quasi-particle lines, each
histogram width."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2005_00827_gb300 import api, inputs

pytestmark = pytest.mark.gpu

# The chord slope (|slope| < 0.3 here) is a sum of FP32 pairs of relative error
# below 1e-5: 3e-6 on Z.  The frequency grid adds the moment expansion's 8^-5.
TOL_Z, TOL_W = 3e-6, 5e-5

GEO = [  # N, nt, nr, tp, propagator, eta
    (4, 2, 2, 0.0, 0, 0.05), (16, 4, 4, 0.0, 0, 0.05),
    (16, 5, 4, -0.2, 0, 0.05), (8, 20, 16, 0.0, 0, 0.05), (24, 2, 10, -0.1, 1, 0.05), (8, 4, 4, 0.0, 0, 0.02),
    (8, 4, 4, -0.2, 0, 0.02), (8, 4, 4, 0.0, 0, 0.0145), (8, 4, 4, 0.0, 0, 0.01)]


def run(N, nt, nr, tp, prop, eta, V, Z, T, w, prec=api.QPFRG_MIXED):
    import torch
    new = lambda *n: torch.full(n, float("nan"), dtype=torch.float64, device="cuda")  # noqa: E731
    with api.Context(N, nt, nr, U=2.0, tp=tp, precision=prec, propagator=prop, eta=eta, n_omega=len(w),
                     omega_min=w[0], omega_max=w[-1]) as c:
        zo, re, im = new(N), new(N, len(w)), new(N, len(w))
        api.qpfrg_selfenergy(c.h, T, torch.from_numpy(V.ravel().copy()).cuda(), torch.from_numpy(Z.copy()).cuda(), re, im, zo)
        torch.cuda.synchronize()
    return zo.cpu().numpy(), re.cpu().numpy() + 1j * im.cpu().numpy()


@pytest.mark.parametrize("kind", ["sym", "asym", "one_entry"])
@pytest.mark.parametrize("geo", GEO, ids=["_".join(map(str, g)) for g in GEO])
def test_selfenergy_targets(geo, kind):
    N, nt, nr, tp, prop, eta = geo
    T, w = 0.2, np.linspace(-3.0, 3.0, 33)
    V = inputs.random_vertex(N, 2.0, seed=N + nt, c4v=kind != "asym")
    Z = inputs.z_profile(N, "aniso")
    if kind == "one_entry":
        V[N // 2, 1, N - 1] *= 1.5
    o = Oracle(N, nt, nr, tp=tp, prop_mode=prop, eta=eta)
    zo, sig = run(N, nt, nr, tp, prop, eta, V, Z, T, w)
    assert np.abs(zo - o.zfactor(T, V, Z)).max() < TOL_Z
    # patches whose sums are their own on every grid (a symmetric vertex copies
    # the others, which differ where momenta lie on a boundary between wedges)
    for j in ((0, N // 4, N // 2) if kind == "sym" else (0, 1, N // 2, N - 1)):
        ref = o.sigma(T, V, Z, j, w)
        assert np.abs(sig[j] - ref).max() < TOL_W * np.abs(ref).max()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_vertex_entry_reaches_its_targets(bad):
    N, T, w = 8, 0.3, np.linspace(-1.0, 1.0, 5)
    V = inputs.random_vertex(N, 2.0, seed=2)
    V[3, 1, 2] = bad
    zo, sig = run(N, 4, 4, 0.0, 0, 0.05, V, np.ones(N), T, w)
    assert np.array_equal(np.isfinite(zo), np.arange(N) != 3)
    assert np.array_equal(np.isfinite(sig).all(axis=1), np.arange(N) != 3) and not np.isfinite(sig[3]).any()


@pytest.mark.parametrize("N,nt,nr", [(8, 4, 4), (16, 8, 6), (8, 32, 16)])
@pytest.mark.parametrize("skew", [0.0, 0.3])
def test_interaction_flow_lines(N, nt, nr, skew):
    """One step from given slopes (skew: not symmetric, every patch evaluated)."""
    import torch
    T, g, dg, w = 0.3, 0.6, 0.05, np.linspace(-2.0, 2.0, 9)
    base = 0.3 + 0.05 * np.cos(8 * np.pi * np.arange(N) / N)
    s1, s2 = -base.copy(), -0.5 * base
    s1[1] -= skew
    out = {}
    for prec in (api.QPFRG_FP64, api.QPFRG_MIXED):
        with api.Context(N, nt, nr, U=2.0, lambda0=g, regulator=api.QPFRG_REG_INTERACTION, T_fixed=T, eta=0.05, step=dg,
                         lambda_end=2.0, sigma_ode=1, z_feedback=1, katanin=1, precision=prec, n_omega=9, omega_min=-2.0,
                         omega_max=2.0) as c:
            img = bytearray(api.qpfrg_get_state(c.h))
            V = inputs.random_vertex(N, 2.0, seed=N)
            tail = np.concatenate([V.ravel(), np.ones(N), s1, s2, np.zeros(4 * N * 9)])
            img[64:] = tail.tobytes()
            api.qpfrg_set_state(c.h, bytes(img))
            api.qpfrg_step(c.h, 1)
            out[prec] = np.frombuffer(api.qpfrg_get_state(c.h)[64:], dtype=np.float64)
    a, b = out[api.QPFRG_MIXED], out[api.QPFRG_FP64]
    n3 = N ** 3
    assert np.abs(a[:n3] - b[:n3]).max() < 1e-5 * np.abs(b[:n3]).max()
    sl, sg = slice(n3 + N, n3 + 3 * N), slice(n3 + 3 * N, None)
    assert np.abs(a[sl] - b[sl]).max() < 1e-5 * np.abs(b[sl]).max()
    assert np.abs(a[sg] - b[sg]).max() < TOL_W * np.abs(b[sg]).max()


# FP64: sums of 1e5 .. 1e7 pairs of relative rounding 1e-15: 1e-12 on Z; the grid's
# moment expansion 8^-5
@pytest.mark.parametrize("kind", ["sym", "asym", "one_entry"])
@pytest.mark.parametrize("geo", [g for g in GEO if g[1] % 2 == 0 and g[1] < 20])
def test_selfenergy_fp64(geo, kind):
    """The FP64 kernel (passes of 128 records, decisions by table)."""
    N, nt, nr, tp, prop, eta = geo
    T, w = 0.2, np.linspace(-3.0, 3.0, 17)
    V = inputs.random_vertex(N, 2.0, seed=N + nt, c4v=kind != "asym")
    Z = inputs.z_profile(N, "aniso")
    if kind == "one_entry":
        V[N // 2, 1, N - 1] *= 1.5
    o = Oracle(N, nt, nr, tp=tp, prop_mode=prop, eta=eta)
    zo, sig = run(N, nt, nr, tp, prop, eta, V, Z, T, w, prec=api.QPFRG_FP64)
    assert np.abs(zo - o.zfactor(T, V, Z)).max() < 1e-12
    for j in (0, 1, N // 2, N - 1):
        ref = o.sigma(T, V, Z, j, w)
        assert np.abs(sig[j] - ref).max() < TOL_W * np.abs(ref).max()


@pytest.mark.parametrize("kind", ["sym", "asym"])
def test_selfenergy_fp64_several_passes(kind):
    """144 loop points per patch (two passes of records); the patches on the
    diagonals, whose pairs lie on no boundary."""
    N, T, w = 8, 0.2, np.linspace(-3.0, 3.0, 9)
    V, Z = inputs.random_vertex(N, 2.0, seed=5, c4v=kind == "sym"), inputs.z_profile(N, "aniso")
    zo, sig = run(N, 12, 12, 0.0, 1, 0.05, V, Z, T, w, prec=api.QPFRG_FP64)
    ref = Oracle(N, 12, 12, prop_mode=1, eta=0.05).zfactor(T, V, Z)
    assert np.abs(zo - ref)[1::2].max() < 1e-12
