"""Calls that meet nuna_shutdown on another thread."""
import threading
import time

import pytest
import torch

from paper_2608_00867_b200 import binding as nb

pytestmark = pytest.mark.gpu


def test_a_call_during_shutdown_waits_and_gets_a_new_context():
    """Shutdown first waits for the device.  A call made meanwhile must not use the context that is about to be freed."""
    nb.nuna_init(1 << 16)
    busy = torch.cuda.Event()
    torch.cuda.synchronize()
    torch.cuda._sleep(2_000_000_000)                       # about a second
    busy.record()
    status = []
    t = threading.Thread(target=lambda: status.append(nb.lib().nuna_shutdown()))
    t.start()
    time.sleep(0.3)                                        # shutdown is waiting for the device by now
    assert not busy.query(), "the device was idle again before the call under test"
    nb.nuna_set_option(nb.NUNA_OPT_PREFETCH, 0)
    assert busy.query(), "the call used a context that shutdown was about to free"
    t.join()
    assert status == [nb.NUNA_OK]
    src = [torch.full((64,), float(r), device="cuda") for r in range(2)]
    dst = [torch.zeros(64, device="cuda") for _ in range(2)]
    nb.nuna_allreduce(src, dst, 64, dtype=nb.NUNA_F32)
    assert all(bool((d == 1.0).all()) for d in dst) and nb.nuna_device_status() == nb.NUNA_OK


def test_the_first_calls_after_shutdown_on_a_stream_of_their_own():
    """A new context's control words, flags and tags are zeroed before a stream that waits for no other may use them: the
    memory may be what an earlier context's last launches wrote, and its epochs start over."""
    n, count = 4, 1 << 20
    src = [torch.full((count,), float(r + 1), device="cuda") for r in range(n)]
    dst = [torch.zeros(count, device="cuda") for _ in range(n)]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(8):
        assert nb.lib().nuna_shutdown() == nb.NUNA_OK
        with torch.cuda.stream(stream):
            for d in dst:
                d.zero_()
            nb.nuna_allreduce_twoshot(src, dst, count, dtype=nb.NUNA_F32)
            nb.nuna_allreduce_twoshot(src, dst, count, dtype=nb.NUNA_F32, flags=nb.NUNA_TWOSHOT_SYS_SCOPE)
        assert nb.nuna_device_status() == nb.NUNA_OK
        assert all(bool((d == 10.0).all()) for d in dst)
