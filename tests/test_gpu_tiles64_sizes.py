"""The FP64 and double-float N^-1 at every tile size, forced by the half-bandwidth: from 2 lambda + 8 > L on a tile of
L samples keeps no output for some block starts and is never taken, and on blocks as few as these the
smallest tile that is left takes least.  Blocks at the edges of its outputs, empty and one-sample blocks:
N^-1 t against the definition, A x and the right-hand side against the oracle, within the FP64-class
operator tolerance (1e-11 of the largest value, as everywhere here)."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from gpu_helpers import cuda, mm, plans, rel_max

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lam,tile", [(2044, 4096), (2045, 8192), (2047, 8192), (4092, 8192), (4093, 16384), (4095, 16384),
                                      (8188, 16384), (8189, 32768), (8190, 32768), (12288, 32768)])
@pytest.mark.parametrize("precision", ["MM_FP64", "MM_DF64"])
def test_forced_tile(precision, lam, tile):
    m = mm()
    keep = (tile - 2 * lam) & ~3
    assert keep >= 8 and (tile == 4096 or tile // 2 - 2 * lam < 8)
    n = min(keep, 4096)
    blocks = [n, 0, n + 1, 1, n - 1, 2 * n + 5, 7, keep, keep + 1 if keep < 9000 else 3]
    prob = synth.random_problem(len(blocks), blocks, 60, lam, seed=lam, gap_frac=0.02, hits_per_pix_min=4)
    if sum(blocks) < 400:   # a few outputs per tile: many tiles would pick a longer one
        assert sum((b + 3) // 4 for b in blocks) <= 152
    gp, op, nb = plans(prob, precision=getattr(m, precision), algo=m.MM_TPLZ_FFT)
    rng = np.random.default_rng(lam)
    x = rng.standard_normal((op.n_obs, 3))
    y = torch.empty(op.n_obs, 3, dtype=torch.float64, device="cuda")
    m.mm_apply_A(gp, cuda(x), y)
    assert rel_max(y.cpu().numpy(), O.apply_A(op, x)) < 1e-11
    m.mm_rhs(gp, cuda(nb["d"]), y)
    assert rel_max(y.cpu().numpy(), O.rhs(op, nb["d"])) < 1e-11
    t = rng.standard_normal(sum(blocks))
    out = torch.empty(sum(blocks), dtype=torch.float64, device="cuda")
    m.mm_apply_Ninv(gp, cuda(t), out)
    assert rel_max(out.cpu().numpy(), O.toeplitz_fft(nb["band"], nb["block_len"], t)) < 1e-11
