"""Ranges of the frequency grid's fixed-point histogram (mixed precision) against
the FP64 call, which bins alike: pole energies outside the bins."""
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
