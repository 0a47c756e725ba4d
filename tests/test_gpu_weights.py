"""The FP64 pointing weights (cos 2 psi, sin 2 psi), read back as P x of unit maps, against extended precision.

Bound: the table's values and the last addition round by 2^-54 each (results below 1), the part that is added
(below 0.05) by less than 2^-57 in its product and sum, and the double-float series by less than 2^-57:
2^-53 + 3 2^-57 = 1.32e-16.  (Forming 1 + (cos r - 1) first costs another rounding: 1.6e-16.)"""
from fractions import Fraction

import numpy as np
import pytest
import torch

from gpu_helpers import mm

pytestmark = pytest.mark.gpu


TWO_PI = Fraction("6.28318530717958647692528676655900576839433879875021")


def reduced(psi):
    """2 psi less the nearest multiple of 2 pi, in extended precision (k times the 43-bit head of 2 pi is exact)."""
    head = Fraction(int(TWO_PI * 2 ** 40), 2 ** 40)
    tail = TWO_PI - head
    tail = np.longdouble(float(tail)) + np.longdouble(float(tail - Fraction(float(tail))))
    x = 2 * psi.astype(np.longdouble)
    k = np.rint(x / np.longdouble(float(TWO_PI)))
    return (x - k * np.longdouble(float(head))) - k * tail


@pytest.mark.parametrize("span", [0.05, 6.3, 300.0, 16000.0])
@pytest.mark.parametrize("precision", ["MM_FP64", "MM_FP32"])
def test_weights(precision, span):
    m = mm()
    n = 1 << 18
    psi = np.random.default_rng(int(span * 100)).uniform(-span, span, n).astype(np.float32)
    pix = torch.arange(n, dtype=torch.int32) % 8
    plan = m.mm_plan(1, 1, [n], 8, pix, torch.from_numpy(psi), 0, torch.ones(1, 1, dtype=torch.float64), cond_max=1e9,
                     precision=getattr(m, precision))
    assert plan.n_obs == 8
    for k, want in ((1, np.cos(reduced(psi))), (2, np.sin(reduced(psi)))):
        x = torch.zeros(8, 3, dtype=torch.float64, device="cuda")
        x[:, k] = 1.0
        t = torch.empty(n, dtype=torch.float64, device="cuda")
        m.mm_apply_P(plan, x, t)
        err = np.abs(t.cpu().numpy().astype(np.longdouble) - want).astype(np.float64)
        assert err.max() < 1.32e-16, err.max()
