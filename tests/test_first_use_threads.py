"""Contexts of several threads that meet a fresh process: each kernel's launch attributes are in place before any
thread launches it."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import threading
import numpy as np
import torch
from paper_1911_12954_gb300 import HOTRG
from workloads import decaying_tensor

torch.zeros(1, device="cuda")
dims, n = (5, 5, 5, 2), 8                      # 9 kept columns: about 100 KB of shared memory a block
T = decaying_tensor(5, dims, 0.7)
ctx = [HOTRG.__new__(HOTRG) for _ in range(n)]
out, gate = [None] * n, threading.Barrier(n)

def work(i):
    gate.wait()
    HOTRG.__init__(ctx[i], batch=1, dcut_max=9, precision="fp16x3", schedule=[(0, 9)], dims0=dims,
                   stream=torch.cuda.Stream())
    ctx[i].set_tensor(T)
    ctx[i].step(0, 9)
    out[i] = ctx[i].tensor()

ts = [threading.Thread(target=work, args=(i,)) for i in range(n)]
[t.start() for t in ts]
[t.join() for t in ts]
assert all(o is not None and np.array_equal(o, out[0]) for o in out)
"""


def test_threads_in_a_fresh_process():
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
