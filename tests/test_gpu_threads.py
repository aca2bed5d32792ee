"""Handles of several threads in a fresh process: the first launches of a kernel come from all of them at once."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = r"""
import threading
import numpy as np
import torch
from paper_1404_2363_gb300.solver import Solver

N = 12
torch.cuda.init()
phi = torch.rand((1200, 1100), device="cuda")
torch.cuda.synchronize()
out, err = [None] * N, []
gate = threading.Barrier(N)

def work(i):
    try:
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            s = Solver(nx=1100, ny=1200, storage=("f32", "bf16")[i % 2], stream=st)
            s.set_D(np.array([[0.03, 0.005], [0.005, 0.04]]))
            s.set_launch(128, (11, 12)[i // 2 % 2])
            s.set_phi(phi)
            gate.wait()
            s.step(12)
            out[i] = s.get_state()[0].cpu()
            s.close()
    except Exception as e:  # noqa: BLE001 - reported below
        err.append(repr(e))
        gate.abort()

ts = [threading.Thread(target=work, args=(i,)) for i in range(N)]
[t.start() for t in ts]
[t.join() for t in ts]
assert not err, err
assert all(torch.equal(out[i], out[i % 2]) for i in range(N))
print("equal")
"""


def test_first_launches_from_several_threads():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "equal" in r.stdout, r.stderr[-2000:]
