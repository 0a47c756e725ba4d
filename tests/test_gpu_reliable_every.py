"""reliable_every up to the largest value of its type asks for no residual replacement before convergence: the
solve takes the iterations and true residuals of one with a merely large value (a replacement after every
iteration, when rounding it to the host's checks overflowed).  Two iterations are allowed for the unordered
FP32 sums, and so is one more true residual where they decide whether the first confirms convergence."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from gpu_helpers import cuda, mm, plans

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def prob():
    return synth.random_problem(3, [1500, 751, 1507], 60, 40, seed=5, gap_frac=0.02, hits_per_pix_min=4, f_knee=20.0,
                                alpha=2.0)


@pytest.mark.parametrize("reliable_every", [2 ** 31 - 1, 2 ** 31 - 5])
@pytest.mark.parametrize("cols", [1, 3])
def test_pcg(prob, reliable_every, cols):
    m = mm()
    gp, op, nb = plans(prob, precision=m.MM_FP32_DF64, algo=m.MM_TPLZ_FFT)
    b = cuda(np.random.default_rng(0).standard_normal((cols, op.n_obs, 3)))

    def solve(every):
        x = torch.empty_like(b)
        info = m.mm_pcg_solve(gp, b, x, tol=1e-6, precision=m.MM_FP32, reliable_every=every)
        return info, x.cpu().numpy()

    large, _ = solve(100000)
    info, x = solve(reliable_every)
    for r in range(cols):
        assert large[r].iters > 4
        assert abs(info[r].iters - large[r].iters) <= 2
        assert info[r].n_true_res <= large[r].n_true_res + 1
        res = b[r].cpu().numpy() - O.apply_A(op, x[r])
        assert np.linalg.norm(res) <= (1e-6 + 1e-9) * float(b[r].norm())


@pytest.mark.parametrize("reliable_every", [2 ** 31 - 1, 2 ** 31 - 3])
def test_server(prob, reliable_every):
    m = mm()
    p = synth.to_numpy(prob)
    srv = m.Server(max_slots=2)

    def solve(every):
        return srv.wait(srv.submit(p["n_det"], 1, p["block_len"].tolist(), p["n_pix"], p["pix"], p["psi"], p["lam"],
                                   p["band"], p["d"], tol=1e-6, reliable_every=every))[1]

    large, info = solve(100000), solve(reliable_every)
    srv.close()
    assert large.iters > 4 and info.status == 0
    assert abs(info.iters - large.iters) <= 2 and info.n_true_res <= large.n_true_res + 1
