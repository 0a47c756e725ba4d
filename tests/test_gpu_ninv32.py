"""The register-transform FP32 N^-1 tiles: A x of FP32 plans against the oracle, within the FP32
operator tolerance (2e-5 of the largest value, as every FP32 A x here), at each tile size the plan
picks (8192, 16384 and 32768 samples: the smallest that holds the band for these few blocks), on
blocks at the edges of a tile's outputs, empty blocks, blocks shorter than the band, odd lengths (so
later blocks start at every alignment), one tile per CTA and several, one column and several."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from gpu_helpers import cuda, mm, plans, rel_max

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile_steps", [0, 3])
@pytest.mark.parametrize("lam,length", [(1, 8192), (600, 8192), (2047, 8192), (4090, 16384), (6000, 16384),
                                        (8190, 32768), (12288, 32768)])
def test_apply_at_tile_edges(lam, length, tile_steps):
    m = mm()
    keep = length - 2 * lam - 4          # outputs of one tile (whatever the block's alignment)
    blocks = [keep, 0, keep + 1, 1, lam + 1, 3 * keep + 5, 7, 2 * keep - 1]
    prob = synth.random_problem(len(blocks), blocks, 150, lam, seed=lam + length, gap_frac=0.02, hits_per_pix_min=4)
    gp, op, _ = plans(prob, precision=m.MM_FP32_DF64, algo=m.MM_TPLZ_FFT, tile_steps=tile_steps)
    rng = np.random.default_rng(lam)
    for cols in (1, 3):
        x = cuda(rng.standard_normal((cols, op.n_obs, 3)))
        y = torch.empty_like(x)
        m.mm_apply_A(gp, x, y)
        for r in range(cols):
            assert rel_max(y[r].cpu().numpy(), O.apply_A(op, x[r].cpu().numpy())) < 2e-5, f"column {r} of {cols}"
