"""What a plan holds per sample: its arrays by type (pixel 4, reduced angle 4, slot 2, weights 8 FP32, 16 FP64 and 16
double-float, sorted entries 2 + 4 + 2 / 32, slots of the groups' pixels) and nothing that only its building needs,
the angles as given (4) among it."""
import pytest
import torch

from gpu_helpers import mm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,per_sample", [("MM_FP64", 4 + 8 + 16), ("MM_DF64", 4 + 2 + 8 + 16 + 16),
                                                  ("MM_FP32", 4 + 4 + 2 + 8 + 16 + 6.0625),
                                                  ("MM_FP32_DF64", 4 + 4 + 2 + 8 + 16 + 16 + 6.0625)])
def test_bytes_per_sample(precision, per_sample):
    m = mm()
    n, n_pix = 1 << 24, 64
    i = torch.arange(n, device="cuda")
    plan = m.mm_plan(1, 1, [n], n_pix, (i % n_pix).int(), (i.double() * 0.37).remainder(3.1).float(), 0,
                     torch.ones(1, 1, dtype=torch.float64, device="cuda"), precision=getattr(m, precision),
                     toeplitz_algo=m.MM_TPLZ_FFT)
    # besides: tables and tiles of at most 2 MB, and 72 + 4 x 64 bytes for each of 1024 to 16384 groups (0.3 B)
    assert per_sample * n <= plan.bytes <= (per_sample + 0.4) * n + (2 << 20), plan.bytes / n
