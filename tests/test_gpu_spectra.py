"""Spectra of many band tables on both sides of the half-bandwidth where their form changes (sum by the definition,
factorised in batches of 256 tables): N^-1 t of 300 blocks with bands of different shapes against the
definition, within the FP64-class operator tolerance (1e-11 of the largest value, as everywhere here)."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_helpers import cuda, mm, rel_max

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lam", [0, 1, 127, 128, 223, 224, 225, 700])
@pytest.mark.parametrize("precision", ["MM_FP64", "MM_FP32_DF64"])
def test_many_tables(precision, lam):
    m = mm()
    nb, n = 300, 260
    rng = np.random.default_rng(lam)
    k = np.arange(lam + 1)
    band = np.stack([np.where(k == 0, 1.0, 0.4 * rng.standard_normal(lam + 1) * np.exp(-k / 5.0) / 5.0) for _ in range(nb)])
    pix, psi = rng.integers(0, 50, nb * n).astype(np.int32), rng.uniform(0, 3, nb * n).astype(np.float32)
    plan = m.mm_plan(nb, 1, [n] * nb, 50, torch.from_numpy(pix), torch.from_numpy(psi), lam,
                     torch.from_numpy(band).contiguous(), precision=getattr(m, precision), toeplitz_algo=m.MM_TPLZ_FFT)
    t = rng.standard_normal(nb * n)
    out = torch.empty(nb * n, dtype=torch.float64, device="cuda")
    m.mm_apply_Ninv(plan, cuda(t), out)
    assert rel_max(out.cpu().numpy(), O.toeplitz_fft(band, np.full(nb, n), t)) < 1e-11
