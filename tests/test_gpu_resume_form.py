"""A flow resumed from its state image takes the form (row orbits or every row) that
the uninterrupted flow takes, and continues it bit for bit."""
import numpy as np
import pytest

from paper_2005_00827_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def steps(c, n):
    """n steps: (state, contraction rows) after each."""
    out = []
    for _ in range(n):
        api.qpfrg_step(c.h, 1)
        out.append((np.frombuffer(api.qpfrg_get_state(c.h)[64:], dtype=np.float64), api.qpfrg_rhs_work(c.h)["contraction_rows"]))
    return out


def both(kw, before, after):
    with api.Context(**kw) as a:
        steps(a, before)
        img = api.qpfrg_get_state(a.h)
        one = steps(a, after)
    with api.Context(**kw) as b:
        api.qpfrg_set_state(b.h, img)
        two = steps(b, after)
    return one, two


@pytest.mark.parametrize("prec", [api.QPFRG_FP64, api.QPFRG_MIXED])
@pytest.mark.parametrize("N,nt,nr,ns,U", [(16, 4, 4, 1, 3.0), (20, 4, 4, 1, 3.0), (32, 2, 4, 1, 4.0), (12, 6, 2, 1, 4.0)])
def test_temperature_flow(N, nt, nr, ns, U, prec):
    one, two = both(dict(N=N, n_theta=nt, n_r=nr, U=U, lambda0=0.4, precision=prec), 20, 3)
    for (va, ra), (vb, rb) in zip(one, two):
        assert ra == rb < N * N
        assert np.array_equal(va, vb)
    V = one[-1][0][:N ** 3].reshape(N, N, N)      # symmetric to the last bit: no tolerance decides
    assert all(np.array_equal(V[np.ix_(g, g, g)], V) for g in map(list, inputs.c4v_patch_maps(N)))


@pytest.mark.parametrize("prec", [api.QPFRG_FP64, api.QPFRG_MIXED, api.QPFRG_MIXED_TC])
@pytest.mark.parametrize("N,nt,nr", [(16, 8, 4), (48, 4, 4)])
def test_interaction_flow(N, nt, nr, prec):
    """The sums of the self-energies are atomic: equal forms, states to rounding."""
    one, two = both(dict(N=N, n_theta=nt, n_r=nr, U=1.5, lambda0=0.0, regulator=api.QPFRG_REG_INTERACTION, T_fixed=0.2,
                         eta=0.05, step=0.05, lambda_end=4.0, sigma_ode=1, z_feedback=1, katanin=1, precision=prec), 3, 2)
    for (va, ra), (vb, rb) in zip(one, two):
        assert ra == rb
        assert np.abs(va - vb).max() < 1e-6 * np.abs(va).max()


@pytest.mark.parametrize("zfb", [0, 1])
@pytest.mark.parametrize("N,nt,nr", [(16, 4, 4), (24, 4, 6), (60, 4, 4)])
def test_tensor_core_flow_keeps_its_symmetry(N, nt, nr, zfb):
    """To the last bit, whatever the order of its atomic sums; Z of the state then needs
    the irreducible targets only."""
    with api.Context(N, nt, nr, U=3.0, lambda0=0.5, precision=api.QPFRG_MIXED_TC, z_feedback=zfb) as c:
        state, rows = steps(c, 6)[-1]
    V, Z = state[:N ** 3].reshape(N, N, N), state[N ** 3:]
    assert rows < N * N
    for g in map(list, inputs.c4v_patch_maps(N)):
        assert np.array_equal(V[np.ix_(g, g, g)], V) and np.array_equal(Z[g], Z)


@pytest.mark.parametrize("off,sym", [(0.2e-5, True), (0.7e-5, True), (0.95e-5, True), (1.2e-5, False), (4e-5, False)])
@pytest.mark.parametrize("entry", [(1, 2, 3), (0, 5, 5)])
def test_image_symmetric_to_the_stated_tolerance(entry, off, sym):
    """A tensor-core state counts as symmetric while every image is within 1e-5 of the
    largest entry, also where a single generator moves an entry by more than a third."""
    N = 16
    with api.Context(N, 4, 4, U=2.0, precision=api.QPFRG_MIXED_TC) as c:
        img = bytearray(api.qpfrg_get_state(c.h))
        V = inputs.random_vertex(N, 2.0, seed=3)
        V[entry] += off * np.abs(V).max()
        img[64:] = np.concatenate([V.ravel(), np.ones(N)]).tobytes()
        api.qpfrg_set_state(c.h, bytes(img))
        api.qpfrg_step(c.h, 1)
        assert (api.qpfrg_rhs_work(c.h)["contraction_rows"] < N * N) == sym
