"""Destroyed plans give all their device memory back: plans of every precision are built, used
(A x, right-hand side, a solve, which allocate on first use) and destroyed several times over, and
the device's free memory must stay where it was after the first round."""
import gc

import pytest
import torch

from gpu_helpers import mm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["MM_FP64", "MM_FP32", "MM_DF64", "MM_FP32_DF64"])
def test_destroyed_plans_return_their_memory(precision):
    m = mm()
    n, side, lam = 1 << 21, 96, 300
    i = torch.arange(n, device="cuda")
    pix = ((i * 7919) % (side * side)).int()
    psi = (i.double() * 0.37).remainder(3.1).float()
    band = torch.zeros(1, lam + 1, dtype=torch.float64, device="cuda")
    band[0, 0], band[0, 1] = 1.0, -0.2
    d = torch.cos(i.double())

    def once():
        gp = m.mm_plan(1, 1, [n], side * side, pix, psi, lam, band, precision=getattr(m, precision))
        b = torch.empty(1, gp.n_obs, 3, dtype=torch.float64, device="cuda")
        m.mm_rhs(gp, d, b)
        x = torch.zeros_like(b)
        m.mm_pcg_solve(gp, b, x, tol=1e-6)
        m.mm_apply_A(gp, b, x)
        del gp
        gc.collect()
        torch.cuda.synchronize()

    once()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(4):
        once()
    # a plan's smallest array of one entry per sample is 4 MB (16-bit slots): four leaks are 16 MB
    assert torch.cuda.mem_get_info()[0] > free - (8 << 20)
