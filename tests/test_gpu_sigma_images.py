"""Frequency grid of a C4v-symmetric vertex in mixed precision, every patch: images
copy their representative's sum, and pairs whose momenta lie on a boundary between
wedges, decided otherwise at the image, are added to it (N not a multiple of 8, odd
n_theta, t' != 0 have them).  Reference: the FP64 call, which sums every patch with
the same decisions (the CPU oracle decides exact ties by the host's rounding)."""
import numpy as np
import pytest

from paper_2005_00827_gb300 import api, inputs

pytestmark = pytest.mark.gpu

# both are binned alike, so that what differs is the FP32 pole energy: 2e-6 of
# error at |E| < 16, against eta = 0.05 at most 4e-5 of a pair
TOL = 5e-5
GEO = [(12, 4, 4, 0.0, 0), (20, 4, 4, 0.0, 0), (16, 5, 4, 0.0, 0), (12, 5, 4, 0.0, 1), (8, 4, 4, -0.2, 0), (4, 3, 2, 0.0, 0),
       (8, 5, 4, -0.2, 1), (48, 5, 4, 0.0, 0), (16, 8, 6, 0.0, 0)]


def sigma(N, nt, nr, tp, prop, prec, V, Z, T, w, eta=0.05):
    import torch
    with api.Context(N, nt, nr, U=2.0, tp=tp, precision=prec, propagator=prop, eta=eta, n_omega=len(w), omega_min=w[0],
                     omega_max=w[-1]) as c:
        re, im = (torch.full((N, len(w)), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2))
        api.qpfrg_selfenergy(c.h, T, torch.from_numpy(V.ravel()).cuda(), torch.from_numpy(Z).cuda(), re, im, None)
        torch.cuda.synchronize()
    return re.cpu().numpy() + 1j * im.cpu().numpy()


def assert_every_patch(got, ref):
    assert (np.abs(got - ref).max(axis=1) < TOL * np.abs(ref).max(axis=1)).all()


@pytest.mark.parametrize("geo", GEO, ids=["_".join(map(str, g)) for g in GEO])
def test_grid_of_every_patch(geo):
    N, nt, nr, tp, prop = geo
    w = np.linspace(-3.0, 3.0, 33)
    V, Z = inputs.random_vertex(N, 2.0, seed=N + nt), inputs.z_profile(N, "aniso")
    ref, got = (sigma(*geo, p, V, Z, 0.2, w) for p in (api.QPFRG_FP64, api.QPFRG_MIXED))
    assert_every_patch(got, ref)


@pytest.mark.parametrize("N,nt,nr,tp", [(12, 4, 4, 0.0), (16, 5, 4, 0.0), (8, 4, 4, -0.2)])
def test_interaction_flow_grid_of_every_patch(N, nt, nr, tp):
    """Sigma and Sigma' after one step from a symmetric state."""
    nw, out = 9, {}
    for prec in (api.QPFRG_FP64, api.QPFRG_MIXED):
        with api.Context(N, nt, nr, U=2.0, tp=tp, lambda0=0.6, regulator=api.QPFRG_REG_INTERACTION, T_fixed=0.2, eta=0.05,
                         step=0.05, lambda_end=2.0, sigma_ode=1, precision=prec, n_omega=nw, omega_min=-2.0,
                         omega_max=2.0) as c:
            img = bytearray(api.qpfrg_get_state(c.h))
            img[64:] = np.concatenate([inputs.random_vertex(N, 2.0, seed=N).ravel(), np.ones(N), np.full(2 * N, -0.05),
                                       np.zeros(4 * N * nw)]).tobytes()
            api.qpfrg_set_state(c.h, bytes(img))
            api.qpfrg_step(c.h, 1)
            y = np.frombuffer(api.qpfrg_get_state(c.h)[64:], dtype=np.float64)[N ** 3 + 3 * N:].reshape(4, N, nw)
            out[prec] = (y[0] + 1j * y[1], y[2] + 1j * y[3])
    for got, ref in zip(out[api.QPFRG_MIXED], out[api.QPFRG_FP64]):
        assert_every_patch(got, ref)
