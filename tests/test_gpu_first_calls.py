"""Calls that come right behind a change of the control words, on a stream that waits for no other."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2608_00867_b200 import binding as nb

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


def test_calls_behind_a_rewind_on_a_stream_of_their_own():
    """A wait that runs out leaves the ticket word rewound by nuna_device_status; the next calls draw from it at once."""
    n, count = 4, 1 << 18
    src = [torch.full((count,), float(r + 1), device="cuda") for r in range(n)]
    dst = [torch.zeros(count, device="cuda") for _ in range(n)]
    stream = torch.cuda.Stream()
    for tagged in (False, True):
        for _ in range(4):
            assert nb.debug_twoshot(src, dst, count, dtype=nb.NUNA_F32, timeout_ms=20, unset_flags=True, tagged=tagged) == nb.NUNA_OK
            assert nb.nuna_device_status() == nb.NUNA_ERR_TIMEOUT
            with torch.cuda.stream(stream):
                for d in dst:
                    d.zero_()
                nb.nuna_allreduce_twoshot(src, dst, count, dtype=nb.NUNA_F32)
                nb.nuna_allreduce_twoshot(src, dst, count, dtype=nb.NUNA_F32, flags=nb.NUNA_TWOSHOT_SYS_SCOPE)
            torch.cuda.synchronize()
            assert all(bool((d == 10.0).all()) for d in dst)
            assert nb.nuna_device_status() == nb.NUNA_OK


def test_the_first_call_with_work_lists_on_a_stream_of_its_own():
    """The lists of a new shape are built and sent during the call that then reads them."""
    flags = nb.NUNA_PLACE_AWARE | nb.NUNA_PLACE_SM_LISTS
    stream = torch.cuda.Stream()
    for n, count in ((4, 8 * 70001), (8, 8 * 30011), (2, 8 * 150007)):
        src = [torch.full((count,), float(r + 1), device="cuda") for r in range(n)]
        dst = [torch.zeros(count, device="cuda") for _ in range(n)]
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            nb.nuna_allreduce_oneshot(src, dst, count, dtype=nb.NUNA_F32, flags=flags)
        torch.cuda.synchronize()
        assert all(bool((d == n * (n + 1) / 2).all()) for d in dst)
    assert nb.nuna_device_status() == nb.NUNA_OK
