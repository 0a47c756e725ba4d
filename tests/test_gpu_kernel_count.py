"""n_kernels counts every kernel of the solve: an FP32 iteration on a plan with pixel windows is P, N^-1, P^T and the
rest of the iteration in one launch (or p, <p, q> and the updates in three when the columns are too many
for it), an FP64 one a tile launch and the rest.  The host looks at the scalars after every iteration here; a
double-float residual takes a handful more."""
import numpy as np
import pytest
import torch

import synth
from gpu_helpers import cuda, mm, plans

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,solve,cols,per", [("MM_FP32_DF64", "MM_FP32", 1, 4), ("MM_FP32_DF64", "MM_FP32", 3, 4),
                                                      ("MM_FP32_DF64", "MM_FP64", 1, 5), ("MM_FP64", "MM_FP64", 1, 2),
                                                      ("MM_FP32_DF64", "MM_FP32", 200, 6)])
def test_iterations_are_counted(precision, solve, cols, per):
    m = mm()
    prob = synth.random_problem(3, [15000, 7510, 15070], 9000, 40, seed=5, hits_per_pix_min=4)
    gp, op, _ = plans(prob, precision=getattr(m, precision), algo=m.MM_TPLZ_FFT)
    b = cuda(np.random.default_rng(0).standard_normal((cols, op.n_obs, 3)))
    x = torch.empty_like(b)
    info = m.mm_pcg_solve(gp, b, x, tol=1e-6, precision=getattr(m, solve), reliable_every=100000, check_every=1)
    it, checks = max(i.iters for i in info), max(i.n_true_res for i in info) + 1
    assert per * it <= info[0].n_kernels <= per * (it + checks) + 10 * checks, (info[0].n_kernels, it, checks)
