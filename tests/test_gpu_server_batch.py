"""More FP32 requests in flight than share a launch of the iteration step (64): every map is the one of the same
problem solved alone, within the accuracy of two solves stopped at 1e-8 (1e-5, as for the other serving tests)."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_helpers import mm

pytestmark = pytest.mark.gpu


def test_many_requests():
    m = mm()
    probs = [synth.to_numpy(synth.random_problem(2, [3001 + 7 * k, 2000], 50 + 13 * k, 30, seed=k, hits_per_pix_min=4,
                                                 f_knee=20.0, alpha=2.0)) for k in range(6)]
    refs = []
    for p in probs:
        op = O.make_plan(p["pix"], p["psi"], p["block_len"], p["band"], p["n_pix"])
        refs.append((op.obs_to_global, O.pcg(op, O.rhs(op, p["d"]), tol=1e-8, max_iter=5000).x))
    srv = m.Server(max_slots=90)
    ids = [srv.submit(p["n_det"], 1, p["block_len"].tolist(), p["n_pix"], p["pix"], p["psi"], p["lam"], p["band"], p["d"],
                      tol=1e-8) for _ in range(20) for p in probs]
    for k, i in enumerate(ids):
        o2g, ref = refs[k % len(probs)]
        mp, info = srv.wait(i)
        assert info.status == 0
        assert np.linalg.norm(mp[o2g] - ref) <= 1e-5 * np.linalg.norm(ref)
    srv.close()
