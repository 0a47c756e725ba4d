"""The FP32 N^-1 of blocks whose bands are multiples of one band: away from a block's ends a constant time
stream comes out as H(0) times the block's scale, and H(0) is small for red noise because the coefficients
of the real-input pair update cancel there.  The scale must not disturb that cancellation: the blocks'
outputs divided by their scales agree.

Four consecutive samples, a quarter turn of 2 psi apart, share a pixel that no other sample sees, and the
map is (1, 0, 0): t = 1 exactly, every frequency but the first is exactly zero, and all inner samples of a
block are one value.  Tolerance: the scale's rounding to FP32, its product, and at most three additions of a
pixel's sum, 2^-24 each, in a block and in the mean it is compared with: 10 2^-24 = 6e-7.  With scaled
coefficients each of the two cancelling ones (about 0.5 each) is rounded on its own: an error near
2^-26 / H(0), 1e-5 and more here."""
import numpy as np
import pytest
import torch

import synth
from gpu_helpers import mm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lam,length", [(700, 80000), (2000, 80000), (8192, 90000)])
def test_scaled_blocks_agree_at_low_frequency(lam, length):
    m = mm()
    n_det = 24
    band, _ = synth.inverse_noise_band(1 << 19, lam, 100.0, 1.0, 1.0, 1.5)
    h0 = float(band[0] + 2 * band[1:].sum())
    assert 0 < h0 < 1e-2 * float(band[0])
    scale = 1.0 / (0.8 + 0.4 * torch.rand(n_det, generator=torch.Generator().manual_seed(1), dtype=torch.float64)) ** 2
    per = length // 4
    i = torch.arange(length)
    pix = (i // 4 + per * torch.arange(n_det)[:, None]).reshape(-1).int()
    psi = ((i % 4).double() * (np.pi / 4)).float().repeat(n_det)
    plan = m.mm_plan(n_det, 1, [length] * n_det, per * n_det, pix.cuda(), psi.cuda(), lam,
                     (band[None] * scale[:, None]).contiguous().cuda(), precision=m.MM_FP32_DF64,
                     toeplitz_algo=m.MM_TPLZ_FFT)
    assert plan.n_obs == per * n_det
    x = torch.zeros(per * n_det, 3, dtype=torch.float64, device="cuda")
    x[:, 0] = 1.0
    y = torch.empty_like(x)
    m.mm_apply_A(plan, x, y)
    edge = (32768 + lam) // 4 + 1   # pixels whose samples' tile, of whatever size, reaches over no end of the block
    got = y[:, 0].reshape(n_det, per)[:, edge:per - edge].cpu().numpy() / 4 / scale.numpy()[:, None]
    assert got.shape[1] > 1000
    # the same H(0) up to its tables' rounding (two numbers near 0.5, 2^-26 each)
    assert abs(got.mean() - h0) < 6e-7 * h0 + 2.0 ** -24, (got.mean(), h0)
    assert np.abs(got / got.mean() - 1.0).max() < 6e-7, np.abs(got / got.mean() - 1.0).max()
