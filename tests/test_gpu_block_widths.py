"""Block CG at the widths where the tall-skinny kernels change their tiling (16, 32 and 64 columns) and
beside them, on a pixel count that is no multiple of any tile: every column against the FP64 PCG of the same
right-hand side, to 1e-5 (the tolerance of the block solves here), with two columns equal so that the pivoted
Cholesky drops a direction."""
import numpy as np
import pytest
import torch

import synth
from gpu_helpers import mm, plans

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [5, 16, 17, 32, 33, 64])
def test_block_widths(width):
    m = mm()
    cfg = synth.tiny_config(n_det=4, n_samp=40000, side=61)
    prob = synth.make_ground_problem(cfg)
    gp, op, nb = plans(prob, precision=m.MM_FP32_DF64)
    rng = np.random.default_rng(width)
    d = np.stack([nb["d"] + rng.standard_normal(nb["d"].size) for _ in range(width)])
    d[-1] = d[0]
    b = torch.empty(width, gp.n_obs, 3, dtype=torch.float64, device="cuda")
    m.mm_rhs(gp, torch.as_tensor(d, device="cuda"), b)
    x, ref = torch.empty_like(b), torch.empty_like(b)
    infos = m.mm_block_cg_solve(gp, b, x, block_width=width, tol=1e-8, max_iter=5000)
    m.mm_pcg_solve(gp, b, ref, tol=1e-10, max_iter=5000, precision=m.MM_FP64)
    assert all(i.status == 0 for i in infos)
    err = (x - ref).flatten(1).norm(dim=1) / ref.flatten(1).norm(dim=1)
    assert float(err.max()) < 1e-5
