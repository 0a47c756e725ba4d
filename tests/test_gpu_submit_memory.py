"""A request larger than the host's memory is refused with MM_ENOMEM (nothing of it is read), and the server goes on:
an exception of the allocator must not cross the C entry, where it would end the process."""
import subprocess
import sys
import os

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import ctypes, numpy as np, torch
import paper_2112_03370_gb300.mm as m
import synth
torch.zeros(1, device="cuda")
srv = m.Server(max_slots=2)
p = synth.to_numpy(synth.random_problem(2, [3001, 2000], 50, 30, seed=1, hits_per_pix_min=4))
args = (p["n_det"], 1, p["block_len"].tolist(), p["n_pix"], p["pix"], p["psi"], p["lam"], p["band"], p["d"])
try:
    srv.submit(p["n_det"], 1, [1 << 58, 2000], *args[3:])
    raise SystemExit("accepted")
except m.MMError as e:
    assert e.code == m.MM_ENOMEM, e.code
mp, info = srv.wait(srv.submit(*args))
assert info.status == 0
srv.close()
print("fine")
"""


def test_request_larger_than_host_memory():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("fine"), (r.returncode, r.stdout, r.stderr[-2000:])
