"""qpfrg_set_state has read the whole image when it returns: a page-locked one may be
overwritten at once (the self-energy ODE's part, here 25 MB, comes last)."""
import pytest

from paper_2005_00827_gb300 import api

pytestmark = pytest.mark.gpu


def test_page_locked_image_may_be_reused_on_return():
    import torch
    N, nw = 48, 16384
    with api.Context(N, 2, 2, U=1.0, lambda0=0.5, regulator=api.QPFRG_REG_INTERACTION, T_fixed=0.3, eta=0.05, step=0.05,
                     lambda_end=2.0, sigma_ode=1, n_omega=nw, omega_min=-1.0, omega_max=1.0) as c:
        head = api.qpfrg_get_state(c.h)[:64]
        body = torch.cat([torch.ones(N ** 3 + N, dtype=torch.float64), torch.arange(2 * N + 4 * N * nw, dtype=torch.float64)])
        img = torch.empty(64 + 8 * body.numel(), dtype=torch.uint8).pin_memory()
        img[:64] = torch.frombuffer(bytearray(head), dtype=torch.uint8)
        img[64:].view(torch.float64).copy_(body)
        tail = img[-4096:]
        for _ in range(3):
            api.qpfrg_set_state_from(c.h, img)
            tail.fill_(255)
            torch.cuda.synchronize()
            img[64:].view(torch.float64).copy_(body)
            sg = torch.zeros(4, N, nw, dtype=torch.float64, device="cuda")
            api.qpfrg_read_sigma_flow(c.h, None, sg, None)
            torch.cuda.synchronize()
            assert torch.equal(sg.cpu().ravel(), body[N ** 3 + 3 * N:])
