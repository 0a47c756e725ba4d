"""One launch per PCG iteration tail (dots, update, next direction) at the sizes where its layout
changes: few pixels (small CTAs), a pixel or two per thread held in registers, more pixels and
columns than fit (loops); one column and several whose iterations end at different times (a zero
right-hand side ends at once, its columns are skipped by P, N^-1 and P^T while the others go on).
Each solution's residual by the oracle must meet the tolerance the solver stopped at (1e-6, plus
1e-9 for the double-float residual it was judged by), with residual replacements in between."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from gpu_helpers import cuda, mm, plans

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reliable_every", [0, 4])
@pytest.mark.parametrize("n_pix,cols", [(1, 1), (150, 1), (150, 4), (9000, 1), (9000, 3), (45000, 1), (45000, 4)])
def test_solutions_meet_the_tolerance(n_pix, cols, reliable_every):
    m = mm()
    n = max(3000, 4 * n_pix)
    prob = synth.random_problem(3, [n, n // 2 + 1, n + 7], n_pix, 40, seed=n_pix + cols, gap_frac=0.02,
                                hits_per_pix_min=4)
    gp, op, _ = plans(prob, precision=m.MM_FP32_DF64, algo=m.MM_TPLZ_FFT)
    b = np.random.default_rng(n_pix).standard_normal((cols, op.n_obs, 3))
    if cols > 1:
        b[1] = 0.0
        b[2] *= 1e-12
    x = torch.zeros(cols, op.n_obs, 3, dtype=torch.float64, device="cuda")
    info = m.mm_pcg_solve(gp, cuda(b), x, tol=1e-6, precision=m.MM_FP32, reliable_every=reliable_every)
    for r in range(cols):
        xr = x[r].cpu().numpy()
        if not b[r].any():
            assert info[r].iters == 0 and not xr.any()
            continue
        res = b[r] - O.apply_A(op, xr)
        assert np.linalg.norm(res) <= (1e-6 + 1e-9) * np.linalg.norm(b[r]), f"column {r} of {cols}"
