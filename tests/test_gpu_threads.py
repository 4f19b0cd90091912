"""Handles of several threads making their first steps at once, in a process where no kernel has run yet.

What a kernel needs before its first launch (its dynamic shared memory, its occupancy) is set up by whichever
thread comes first; the others must find it done.  Eight threads wait at a barrier, then each steps a chain of
its own (reductions above 64 rows, all three engines); every thread has to succeed, and threads with the same
inputs have to end bitwise equal.  Each process gives the race one chance, so there are four.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """
import threading
import numpy as np
import workloads
from paper_2401_05301_gb300 import TEBD
B, lam, _ = workloads.synthetic_state(8, 4, 24)
sims = []
for k in range(8):
    g = TEBD(8, 3, 24, 4.0, 1.0, 0.1, 0.004, 4.5, 0.02, precision=k % 3)
    g.set_state(B, lam)
    sims.append(g)
gate, errors = threading.Barrier(8), []
def first_step(g):
    gate.wait()
    try:
        g.step(1)
    except Exception as e:
        errors.append(e)
threads = [threading.Thread(target=first_step, args=(g,)) for g in sims]
for t in threads: t.start()
for t in threads: t.join()
assert not errors, errors
out = [g.measure()[0] for g in sims]
for k in range(3, 8):
    assert np.array_equal(out[k], out[k - 3]), k
"""


@pytest.mark.parametrize("attempt", range(4))
def test_first_steps_at_once(lib, attempt):
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-2000:]
