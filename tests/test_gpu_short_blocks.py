"""Blocks far shorter than the band at the half-bandwidths where 2 lambda + 6 is a tile length (4096, 8192
and 16384 samples): a tile of that length keeps no output for some block starts, so the plan has to take
the next longer one.  (Choosing it all the same divided by zero on the host.)  A x and the right-hand side
against the oracle, within the operators' tolerances."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from gpu_helpers import cuda, mm, plans, rel_max

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lam", [2045, 4093, 8189])
@pytest.mark.parametrize("precision,tol", [("MM_FP64", 1e-11), ("MM_DF64", 1e-11), ("MM_FP32_DF64", 2e-5)])
def test_band_leaves_a_tile_without_outputs(precision, tol, lam):
    m = mm()
    blocks = [100, 131, 0, 1, 50]
    prob = synth.random_problem(len(blocks), blocks, 12, lam, seed=lam, hits_per_pix_min=4)
    gp, op, nb = plans(prob, precision=getattr(m, precision))
    x = np.random.default_rng(lam).standard_normal((op.n_obs, 3))
    y = torch.empty(op.n_obs, 3, dtype=torch.float64, device="cuda")
    m.mm_apply_A(gp, cuda(x), y)
    assert rel_max(y.cpu().numpy(), O.apply_A(op, x)) < tol
    m.mm_rhs(gp, cuda(nb["d"]), y)
    assert rel_max(y.cpu().numpy(), O.rhs(op, nb["d"])) < 1e-11
