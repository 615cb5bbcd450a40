"""The student's first step in threads that have made no CUDA call yet (needs a
GB300)."""
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


_FIRST_USE = """
import threading
import numpy as np, torch
from paper_2601_01903_gb300 import student
torch.zeros(1, device="cuda")
params = student.init_params(8, 128, 37, 0)
students = [student.Student(8, 128, 37, 64, params) for _ in range(16)]
x, labels = torch.zeros(64, 8, device="cuda"), torch.zeros(64, 37, device="cuda")
target = torch.zeros(64, device="cuda")
torch.cuda.synchronize()
go, failed = threading.Barrier(16), []
def first(s):
    go.wait()
    try:
        s.gradients(x, labels, target, 0.0)
    except Exception as e:
        failed.append(e)
threads = [threading.Thread(target=first, args=(s,)) for s in students]
[t.start() for t in threads]
[t.join() for t in threads]
torch.cuda.synchronize()
assert not failed, failed
"""


def test_first_use_from_several_threads_at_once():
    """The tensor maps are made on the first step of a student, by an encoder that
    wants a current context; it is looked up on the first step of a process."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _FIRST_USE], capture_output=True, text=True, timeout=200, cwd=root)
    assert r.returncode == 0, r.stderr[-2000:]
