"""The first plans of a process, made by many threads at once: what the device can hold is asked for once and kept, and a
thread that comes while another asks gets the same plan as one that comes later."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))

PROGRAM = """
import threading
import torch
from paper_2410_11744_b200 import binding as B
torch.cuda.init()
for regime, n, d in ((0, 64, 128), (0, 64, 64), (1, 256, 128), (1, 256, 64)):
    B.dyspec_set_tuning(regime, 0, 2)
    gate, got = threading.Barrier(16), [None] * 16
    def make(k):
        torch.cuda.set_device(0)
        gate.wait()
        got[k] = B.Plan(32, 32, d, [1024], [n], [0], 1024 + n, B.dyspec_words_per_row(n), 0.0).describe()
    threads = [threading.Thread(target=make, args=(k,)) for k in range(16)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    later = B.Plan(32, 32, d, [1024], [n], [0], 1024 + n, B.dyspec_words_per_row(n), 0.0).describe()
    assert later["cluster"] > 1, later
    assert all(g == later for g in got), (later, got)
"""


def test_threads_that_come_first_get_the_plan_that_later_ones_get():
    env = dict(os.environ, PYTHONPATH=os.path.dirname(HERE))
    r = subprocess.run([sys.executable, "-c", PROGRAM], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
