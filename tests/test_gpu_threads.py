"""Handles on several host threads, each with a stream of its own: the first
launches of a process, which look up what the device holds, among them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import ctypes, threading
import numpy as np, torch
from paper_1003_3779_gb300 import inputs, qw
jobs = [((600, 520), inputs.grover(), 0), ((300, 200), inputs.grover(), 1), ((9001,), inputs.su2(0.3), 0), ((700, 700), inputs.hadamard2(), 2)]
psi = [inputs.random_state((2 * len(d),) + tuple(reversed(d)), seed=i, dtype=np.complex64) for i, (d, _, _) in enumerate(jobs)]
torch.cuda.init()
got, gate = [None] * 16, threading.Barrier(16)
def go(i):
    d, C, shift = jobs[i % 4]
    s = torch.cuda.Stream()
    w = qw.Walk(d, prec="f32", shift=shift, stream=ctypes.c_void_p(s.cuda_stream)).set_coin(C)
    if len(d) == 1:
        w.set_plan_ex(512, 256, 2)
    gate.wait()
    got[i] = w.set_state(psi[i % 4]).step(200).state(np.complex64)
    w.close()
threads = [threading.Thread(target=go, args=(i,)) for i in range(16)]
[t.start() for t in threads]
[t.join() for t in threads]
for i in range(4, 16):
    assert np.array_equal(got[i], got[i % 4]), i
for i, (d, C, shift) in enumerate(jobs):
    w = qw.Walk(d, prec="f32", shift=shift).set_coin(C)
    if len(d) == 1:
        w.set_plan_ex(512, 256, 2)
    assert np.array_equal(got[i], w.set_state(psi[i]).step(200).state(np.complex64)), i
print("same")
"""


def test_first_launches_from_many_threads():
    for _ in range(3):
        p = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300)
        assert p.returncode == 0 and p.stdout.strip() == "same", p.stderr[-2000:]
