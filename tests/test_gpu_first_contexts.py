"""A process's first contexts may be created by several threads at once (a context
belongs to one thread, the rule tables on the device to all of them): every thread
gets a context whose results are those of a context created alone."""
import subprocess
import sys
import os

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import threading
import torch
from paper_1610_09991_gb300 import paid as P, workloads as W
lm = torch.as_tensor(W.all_pairs(9), dtype=torch.int32, device="cuda")
q = torch.as_tensor(W.q_grid_bz(2), device="cuda")
P.load()
N, gate, got = 8, threading.Barrier(8), [None] * 8
modes = [dict(), dict(eval_fp32=1, rule_n=6), dict(group_mode=1, rule_n=12),
         dict(group_mode=1, rule_n=12, eval_fp32=1)]
def one(i, wait=True):
    if wait:
        gate.wait()
    ctx = P.Context(*W.LATTICE, ffset=9, **modes[i % 4])
    with torch.cuda.stream(torch.cuda.Stream()):
        r = ctx.integrate_batch(P.PH, q, lm, 0.3, 1e-5)
        torch.cuda.current_stream().synchronize()
    ctx.close()
    return [x.cpu() for x in (r.values, r.errors, r.regions, r.status)]
def run(i):
    got[i] = one(i)
torch.cuda.synchronize()
ts = [threading.Thread(target=run, args=(i,)) for i in range(N)]
[t.start() for t in ts]
[t.join() for t in ts]
for i in range(N):
    assert got[i] is not None, i
    for a, b in zip(got[i], one(i, False)):
        assert torch.equal(a, b), i
print("same")
"""


def test_threads_that_create_the_first_contexts_together():
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True,
                           timeout=300)
        assert r.returncode == 0 and r.stdout.strip() == "same", r.stdout + r.stderr
