"""The tuner times the plan's own choices beside its candidates, so that what it keeps was at least as fast: a
small plan's 1024-sample window groups, and the tiles that a CTA walks (a walk of 3 is no candidate of the
tuner's own).  The tuned operator matches the oracle (FP32 tolerance of the parity tests)."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from gpu_helpers import cuda, mm, plans, rel_max

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile_steps", [0, 3])
def test_own_choices_are_timed(tile_steps):
    m = mm()
    prob = synth.make_ground_problem(synth.tiny_config(n_det=4, n_samp=65536))
    gp, op, _ = plans(prob, precision=m.MM_FP32_DF64, tile_steps=tile_steps)
    res = m.mm_autotune(gp, max_width=2)
    assert 1024 in res["win_ms"]
    assert (tile_steps or 1) in res["steps_ms"]
    assert res["win_ms"][res["win_samples"]] == min(res["win_ms"].values())
    assert res["steps_ms"][res["tile_steps"]] == min(res["steps_ms"].values())
    assert res["n_rejected"] == 0
    x = np.random.default_rng(1).standard_normal((op.n_obs, 3))
    y = torch.empty(op.n_obs, 3, dtype=torch.float64, device="cuda")
    m.mm_apply_A(gp, cuda(x), y)
    assert rel_max(y.cpu().numpy(), O.apply_A(op, x)) < 2e-5
