"""FP32 P^T on plans whose pixels get many additions: they are spread over several maps.

Rounding error of a sum of n positive unequal terms (the map's polarisation varies with the angle; equal
terms would round alike) added one after the other to an FP32 map: each addition rounds by ulp / sqrt(12) of
the sum so far, whose ulp is 2^-24 to 2^-23 of it (rms over a binade 1.44 2^-24), so the relative rms error
is 1.44 2^-24 sqrt(n / 36).  Here a pixel gets 160 additions: 1.8e-7 in one map; in four
maps 40 each, 4.5e-8, and three more additions of the maps, 3.3e-8: 5.6e-8 together.  The bound of 1e-7
lies between the two, 1.8 times from each."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from gpu_helpers import cuda, mm, plans, rel_max

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols", [1, 3])
@pytest.mark.parametrize("pt_sub", [0, 4096])
def test_rounding_of_many_additions(pt_sub, cols):
    m = mm()
    n, n_pix, dwell = 1 << 21, 2048, 8
    rng = np.random.default_rng(3)
    pix = np.repeat(rng.permutation(np.repeat(np.arange(n_pix), n // dwell // n_pix)), dwell).astype(np.int32)
    psi = rng.uniform(0, 3, n).astype(np.float32)
    plan = m.mm_plan(1, 1, [n], n_pix, torch.from_numpy(pix).cuda(), torch.from_numpy(psi).cuda(), 0,
                     torch.ones(1, 1, dtype=torch.float64, device="cuda"), precision=m.MM_FP32_DF64, pt_sub=pt_sub)
    assert plan.n_obs == n_pix
    x = np.zeros((cols, n_pix, 3))
    x[:, :, 0] = rng.uniform(1, 2, (cols, n_pix))
    x[:, :, 1:] = rng.uniform(-0.3, 0.3, (cols, n_pix, 2))
    x = x.astype(np.float32).astype(np.float64)
    y = torch.empty(cols, n_pix, 3, dtype=torch.float64, device="cuda")
    m.mm_apply_A(plan, cuda(x), y)
    c, s = np.cos(2.0 * psi.astype(np.float64)), np.sin(2.0 * psi.astype(np.float64))
    for r in range(cols):   # N^-1 = 1: the intensity entry of P^T P x is the sum of the pixel's samples
        t = x[r, pix, 0] + c * x[r, pix, 1] + s * x[r, pix, 2]
        err = y[r, :, 0].cpu().numpy() / np.bincount(pix, weights=t, minlength=n_pix) - 1.0
        assert np.sqrt((err ** 2).mean()) < 1e-7, np.sqrt((err ** 2).mean())


@pytest.mark.parametrize("n_pix,cols,pt_sub", [(40, 1, 0), (100, 5, 0), (100, 3, 8192), (700, 2, 0)])
def test_operator_and_solve(n_pix, cols, pt_sub):
    """A x against the oracle and a solve whose columns end at different times."""
    m = mm()
    prob = synth.random_problem(3, [50001, 30000, 40007], n_pix, 40, seed=n_pix, gap_frac=0.02, hits_per_pix_min=4)
    gp, op, _ = plans(prob, precision=m.MM_FP32_DF64, algo=m.MM_TPLZ_FFT, pt_sub=pt_sub)
    rng = np.random.default_rng(n_pix)
    x = rng.standard_normal((cols, op.n_obs, 3))
    y = torch.empty(cols, op.n_obs, 3, dtype=torch.float64, device="cuda")
    m.mm_apply_A(gp, cuda(x), y)
    for r in range(cols):
        assert rel_max(y[r].cpu().numpy(), O.apply_A(op, x[r])) < 2e-5
    b = rng.standard_normal((cols, op.n_obs, 3))
    if cols > 1:
        b[1] = 0.0
    xs = torch.empty(cols, op.n_obs, 3, dtype=torch.float64, device="cuda")
    m.mm_pcg_solve(gp, cuda(b), xs, tol=1e-6, precision=m.MM_FP32)
    for r in range(cols):
        res = b[r] - O.apply_A(op, xs[r].cpu().numpy())
        assert np.linalg.norm(res) <= (1e-6 + 1e-9) * np.linalg.norm(b[r])


def test_server_requests():
    """Requests of plans with one and with several maps side by side."""
    m = mm()
    probs = [synth.random_problem(2, [50001, 40007], n_pix, 40, seed=n_pix, hits_per_pix_min=4) for n_pix in (60, 9000, 250)]
    srv = m.Server(max_slots=4)
    nb = [synth.to_numpy(p) for p in probs]
    ids = [srv.submit(p["n_det"], 1, p["block_len"].tolist(), p["n_pix"], p["pix"], p["psi"], p["lam"], p["band"],
                      p["d"], tol=1e-8) for p in nb]
    out = [srv.wait(i) for i in ids]
    srv.close()
    for p, (mp, info) in zip(nb, out):
        op = O.make_plan(p["pix"], p["psi"], p["block_len"], p["band"], p["n_pix"])
        ref = O.pcg(op, O.rhs(op, p["d"]), tol=1e-8, max_iter=5000).x
        assert info.status == 0
        assert np.linalg.norm(mp[op.obs_to_global] - ref) <= 1e-5 * np.linalg.norm(ref)
