"""MM_TPLZ_AUTO on blocks short enough for the tensor-core product and on longer ones, around the half-bandwidths
where its estimate changes (0, 32, 64): A x and the right-hand side against the oracle (the FP32 tolerance
of the parity tests, 1e-11 for the double-float right-hand side), several columns, ragged and empty blocks."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from gpu_helpers import cuda, mm, plans, rel_max

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lam", [0, 1, 32, 33, 64, 65])
@pytest.mark.parametrize("blocks", [[37, 0, 100, 61, 256, 1] * 8, [4096, 4097, 1000, 8192], [30000, 9]])
def test_auto_matches_oracle(blocks, lam):
    m = mm()
    prob = synth.random_problem(len(blocks), blocks, 60, lam, seed=lam + len(blocks), gap_frac=0.02, hits_per_pix_min=4)
    gp, op, nb = plans(prob, precision=m.MM_FP32_DF64, algo=m.MM_TPLZ_AUTO)
    x = np.random.default_rng(lam).standard_normal((3, op.n_obs, 3))
    y = torch.empty(3, op.n_obs, 3, dtype=torch.float64, device="cuda")
    m.mm_apply_A(gp, cuda(x), y)
    for r in range(3):
        assert rel_max(y[r].cpu().numpy(), O.apply_A(op, x[r])) < 2e-5
    b = torch.empty(op.n_obs, 3, dtype=torch.float64, device="cuda")
    m.mm_rhs(gp, cuda(nb["d"]), b)
    assert rel_max(b.cpu().numpy(), O.rhs(op, nb["d"])) < 1e-11
