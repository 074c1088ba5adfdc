"""Batched flows whose Runge-Kutta state lives on the representative rows: patch
counts with partly filled blocks and mirror-line pairs, every channel alone and all
together, and several flows of which some stop on the way, against the same flows
run alone on all elements."""
import pytest

from paper_2005_00827_gb300 import api

pytestmark = pytest.mark.gpu

# the two paths round FP32 stage vertices alike and add the FP32 partial sums of the
# tensor-core contraction in other orders: 1e-6 of a stage's dV each (2^-20 per sum),
# random over the 40 x 4 stages of a flow
REL = 2e-5


@pytest.mark.parametrize("mask", [1, 2, 4, 7])
@pytest.mark.parametrize("N,nt,nr", [(8, 2, 2), (16, 4, 4), (24, 2, 4), (40, 3, 2), (96, 2, 2), (104, 4, 2)])
def test_batch_rows_match_single_flows(N, nt, nr, mask):
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    kw = dict(precision=api.QPFRG_MIXED_TC, channel_mask=mask, max_steps=40)
    o = api.qpfrg_default_options()
    for k, v in kw.items():
        setattr(o, k, v)
    specs = [(N, 1.5, 0.5, 0.01), (N, 3.0, 0.5, 0.3), (N, 2.25, 0.5, 0.24)]
    res = api.qpfrg_flow_batch(api.qpfrg_lattice(1.0, 0.0, 0.0), api.qpfrg_fine_grid(nt, nr, 0),
                               api.QPFRG_REG_TEMPERATURE, o, specs, stream)
    for (n, U, T0, Tend), r in zip(specs, res):
        with api.Context(n, nt, nr, U=U, lambda0=T0, lambda_end=Tend, stream=stream, **kw) as c:
            one = api.qpfrg_flow(c.h).as_dict()
        assert (r["status"], r["steps"]) == (one["status"], one["steps"])
        assert r["lam"] == pytest.approx(one["lam"], rel=1e-12)
        assert r["max_abs_v"] == pytest.approx(one["max_abs_v"], rel=REL)
