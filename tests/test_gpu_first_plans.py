"""The first plans of a process, built and used by several threads at once on streams of their own: no launch may come
before its kernel's shared-memory limit is set.  Every thread's A x equals that of a plan built afterwards, up to
the order of FP64 sums."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import threading, torch
import paper_2112_03370_gb300.mm as m
import synth
prob = synth.random_problem(2, [30001, 20000], 50, 300, seed=1, hits_per_pix_min=4)
pix, psi, band = prob.pix.cuda(), prob.psi.cuda(), prob.band.cuda()
torch.cuda.synchronize()
gate, out, n = threading.Barrier(8), {}, 8

def use(k):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        gate.wait()
        plan = m.mm_plan(2, 1, prob.block_len.tolist(), 50, pix, psi, prob.lam, band,
                         precision=(m.MM_FP64, m.MM_FP32_DF64)[k % 2])
        x = torch.ones(plan.n_obs, 3, dtype=torch.float64, device="cuda")
        y = torch.empty_like(x)
        m.mm_apply_A(plan, x, y)
        stream.synchronize()
        out[k] = y

ts = [threading.Thread(target=use, args=(k,)) for k in range(n)]
[t.start() for t in ts]
[t.join() for t in ts]
assert len(out) == n, sorted(out)
first, gate = dict(out), threading.Barrier(1)
for k in range(2):
    use(k)   # again, alone
for k in range(n):
    ref = out[k % 2]
    assert float((first[k] - ref).abs().max()) <= (1e-12 if k % 2 == 0 else 2e-5) * float(ref.abs().max()), k
print("fine")
"""


def test_threads_build_the_first_plans():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE], cwd=root, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("fine"), (r.returncode, r.stdout, r.stderr[-3000:])
