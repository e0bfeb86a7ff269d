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
