"""Calls that come right behind a change of the control words, on a stream that waits for no other."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_first_static_call_of_a_process_on_a_stream_of_its_own():
    """In a fresh process: three calls in a row, of which the first finds the fixed arrays as the library's load left them."""
    code = """
import torch
from paper_2608_00867_b200 import binding as nb
n, count = 4, 1 << 20
src = [torch.full((count,), float(r + 1), device="cuda") for r in range(n)]
dst = [[torch.zeros(count, device="cuda") for _ in range(n)] for _ in range(3)]
torch.cuda.synchronize()
with torch.cuda.stream(torch.cuda.Stream()):
    for d in dst:
        nb.nuna_allreduce_twoshot_static(src, d, count, dtype=nb.NUNA_F32)
torch.cuda.synchronize()
assert all(bool((t == 10.0).all()) for d in dst for t in d)
assert nb.nuna_device_status() == nb.NUNA_OK
"""
    done = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stderr[-2000:]
