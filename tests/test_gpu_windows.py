"""P and P^T of the FP32 A-application over the pixel windows at the edges of their layouts: A x
against the oracle within the FP32 operator tolerance (2e-5 of the largest value), for one pixel (a
single run through every lane's entries), few and more pixels than a window holds (groups are split
down), many short rows (fewer samples than a lane's entries) and few long ones, rows at every
alignment, empty rows, flagged samples, one column and several; and the same operator rebuilt by the
autotuner over every group size."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from gpu_helpers import cuda, mm, plans, rel_max

pytestmark = pytest.mark.gpu

SHAPES = {
    "few long rows": [40001, 40003, 39998],
    "one row": [70001],
    "many short rows": [33 + (7 * i) % 31 for i in range(600)],
    "short and empty rows": [(97 * i) % 300 for i in range(130)],
    "rows around a window": [1024, 1023, 1025, 2047, 2049, 31, 32, 33, 1, 0],
}


@pytest.mark.parametrize("n_pix", [1, 40, 9000])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_apply_over_windows(shape, n_pix):
    m = mm()
    blocks = SHAPES[shape]
    n_pix = min(n_pix, max(1, sum(blocks) // 8))
    prob = synth.random_problem(len(blocks), blocks, n_pix, 3, seed=n_pix + len(blocks), gap_frac=0.05,
                                hits_per_pix_min=4)
    gp, op, _ = plans(prob, precision=m.MM_FP32_DF64, algo=m.MM_TPLZ_FFT)
    rng = np.random.default_rng(n_pix)
    x = cuda(rng.standard_normal((3, op.n_obs, 3)))
    ref = [O.apply_A(op, x[r].cpu().numpy()) for r in range(3)]
    for cols in (1, 3):
        y = torch.empty_like(x[:cols])
        m.mm_apply_A(gp, x[:cols].contiguous(), y)
        for r in range(cols):
            assert rel_max(y[r].cpu().numpy(), ref[r]) < 2e-5, f"column {r} of {cols}"
    tune = m.mm_autotune(gp, max_width=1)   # rebuilds the windows at every group size
    assert tune["n_rejected"] == 0 and tune["max_rel_dev"] < 2e-5
    y = torch.empty_like(x[0])
    m.mm_apply_A(gp, x[0].contiguous(), y)
    assert rel_max(y.cpu().numpy(), ref[0]) < 2e-5
