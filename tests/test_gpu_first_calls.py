"""The first calls of a process from several threads at once: each must find what the library sets
up on first use (the tensor-map encoder, kernel attributes) complete, not half set up by another
thread.  In a process of its own, so that these are first calls."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import threading
import torch
from paper_2201_06914_gb300 import wp
n, cnt, N, r = 16, 64, 203, 8
jobs = []
for i in range(n):
    g = torch.Generator(device="cuda").manual_seed(i)
    A, Q = torch.randn(1, cnt, N, generator=g, device="cuda"), torch.randn(1, cnt, r, generator=g, device="cuda")
    jobs.append((A, Q, torch.zeros(1, r, N, device="cuda"), wp.workspace(wp.wp_probe_accumulate_workspace_bytes(1, cnt, r)),
                 torch.cuda.Stream()))
torch.cuda.synchronize()
start, errors = threading.Barrier(n), []
def call(A, Q, P, ws, s):
    start.wait()
    try:
        wp.wp_probe_accumulate(A, cnt, N, 1, Q, cnt, 0, r, 1.0, P, ws, stream=s)
    except Exception as e:
        errors.append(str(e))
threads = [threading.Thread(target=call, args=j) for j in jobs]
[t.start() for t in threads]
[t.join() for t in threads]
torch.cuda.synchronize()
assert not errors, errors
for A, Q, P, ws, s in jobs:
    ref = Q[0].double().T @ A[0].double()
    assert ((P[0].double() - ref).norm() / ref.norm()).item() < 1e-5
"""


def test_first_calls_from_many_threads():
    p = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
