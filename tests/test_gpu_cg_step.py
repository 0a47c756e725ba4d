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


def test_columns_replaced_at_other_times_leave_a_column_alone():
    """A column's search directions do not depend on when the other columns pause for their residual
    replacement.  Right-hand sides made of m eigenvectors of M A end after about m iterations, so the
    first column iterates beside up to eight replacements of the others; forming its next direction
    again at each of them takes it from 10 iterations to more than 100 (dense CG in 64 bits, which
    FP32-sized errors in A p change by no iteration).  Two are allowed for the order of FP32 sums."""
    m = mm()
    prob = synth.random_problem(3, [1500, 751, 1507], 60, 40, seed=5, gap_frac=0.02, hits_per_pix_min=4,
                                f_knee=20.0, alpha=2.0)
    gp, op, _ = plans(prob, precision=m.MM_FP32_DF64, algo=m.MM_TPLZ_FFT)
    n = 3 * op.n_obs
    A = np.stack([O.apply_A(op, e.reshape(-1, 3)).ravel() for e in np.eye(n)], 1)
    L = np.zeros((n, n))
    for i in range(op.n_obs):
        L[3 * i:3 * i + 3, 3 * i:3 * i + 3] = np.linalg.cholesky(op.Minv[i])
    V = np.linalg.eigh(L.T @ (0.5 * (A + A.T)) @ L)[1]
    b = [np.random.default_rng(0).standard_normal(n)]
    for k in (1, 2, 3, 4, 5, 6, 7, 8):
        b.append(np.linalg.solve(L.T, V[:, np.linspace(0, n - 1, k).astype(int)].sum(axis=1)))
    b = np.array(b).reshape(len(b), op.n_obs, 3)

    def iters(cols):
        x = torch.zeros(len(cols), op.n_obs, 3, dtype=torch.float64, device="cuda")
        info = m.mm_pcg_solve(gp, cuda(cols), x, tol=1e-6, max_iter=500, precision=m.MM_FP32, check_every=1)
        return [i.iters for i in info]

    alone, together = iters(b[:1]), iters(b)
    assert len(set(together)) >= 4, together
    assert together[0] <= alone[0] + 2, (alone, together)
