"""The FP64 and double-float N^-1 tiles at each size a plan picks (4096 to 32768 samples), on blocks at
the edges of a tile's outputs, empty blocks, blocks shorter than the band and odd lengths: N^-1 t against
the definition, A x and the right-hand side against the oracle, within the FP64-class operator tolerance
(1e-11 of the largest value, as everywhere here)."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from gpu_helpers import cuda, mm, plans, rel_max

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lam,length", [(1, 4096), (700, 4096), (1500, 8192), (3000, 16384), (4094, 16384),
                                        (7000, 32768)])
@pytest.mark.parametrize("precision", ["MM_FP64", "MM_DF64"])
def test_tiles_at_edges(precision, lam, length):
    m = mm()
    keep = length - 2 * lam - 4
    blocks = [keep, 0, keep + 1, 1, lam + 1, 3 * keep + 5, 7, 2 * keep - 1]
    prob = synth.random_problem(len(blocks), blocks, 150, lam, seed=lam, gap_frac=0.02, hits_per_pix_min=4)
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
