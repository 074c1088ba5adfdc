"""Input differences of a few 1e-7 in mixed precision (several units of FP32) are
computed, not dropped with the symmetry: Z of a given vertex, and the flows' right-hand
sides from a state image."""
import numpy as np
import pytest

from paper_2005_00827_gb300 import api, inputs

pytestmark = pytest.mark.gpu

N = 16


def z_of(prec, V, Z):
    import torch
    with api.Context(N, 4, 4, U=2.0, precision=prec, eta=0.05) as c:
        out = torch.zeros(N, dtype=torch.float64, device="cuda")
        api.qpfrg_selfenergy(c.h, 0.2, torch.from_numpy(V.ravel()).cuda(), torch.from_numpy(Z).cuda(), None, None, out)
        torch.cuda.synchronize()
    return out.cpu().numpy()


def test_z_of_a_vertex_that_is_symmetric_but_for_3e7():
    """The rows of patch 1 scaled by 1 + 3e-7: its Z moves from its image's, patch 3, by
    2 x 3e-7 of its slope.  Both are FP32 sums of the same pairs; what the rounding of
    the scaled entries (6e-8 each, independent) leaves is a tenth of that."""
    V, Z = inputs.random_vertex(N, 6.0, seed=3), inputs.z_profile(N, "aniso")
    V[1] *= 1.0 + 3e-7 * 0.99
    d = {p: (lambda z: z[1] - z[3])(z_of(p, V, Z)) for p in (api.QPFRG_FP64, api.QPFRG_MIXED)}
    assert abs(d[api.QPFRG_MIXED] - d[api.QPFRG_FP64]) < 0.5 * abs(d[api.QPFRG_FP64])


@pytest.mark.parametrize("kind", ["temperature", "interaction"])
def test_flow_state_that_is_symmetric_but_for_1e7(kind):
    V = inputs.random_vertex(N, 2.0, seed=3)
    tail = [V.ravel(), np.ones(N)]
    kw = dict(U=2.0, precision=api.QPFRG_MIXED)
    if kind == "interaction":
        kw.update(lambda0=0.5, regulator=api.QPFRG_REG_INTERACTION, T_fixed=0.2, eta=0.05, step=0.05, lambda_end=4.0,
                  sigma_ode=1, z_feedback=1)
        s1 = np.full(N, -0.1)
        s1[3] *= 1.0 + 2e-7          # 2e-8 of Z
        tail += [s1, np.zeros(N)]
    else:
        kw.update(lambda0=0.5)
        V[1, 2, 3] += 9e-8 * np.abs(V).max()
        tail[0] = V.ravel()
    with api.Context(N, 4, 4, **kw) as c:
        img = bytearray(api.qpfrg_get_state(c.h))
        img[64:] = np.concatenate(tail).tobytes()
        api.qpfrg_set_state(c.h, bytes(img))
        api.qpfrg_step(c.h, 1)
        assert api.qpfrg_rhs_work(c.h)["contraction_rows"] == N * N
