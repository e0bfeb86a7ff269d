"""Stream order of eagerly issued calls without any launch flag, among each other and with torch's own kernels."""
import pytest
import torch

from paper_2608_00867_b200 import binding as nb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side_stream", [False, True])
@pytest.mark.parametrize("count", [8, 2049, 70001])
def test_unflagged_calls_keep_stream_order(count, side_stream):
    """torch writes the sources, one-shot -> two-shot (flags, put) -> alltoall -> reduce-scatter -> allgather each read
    what the call before wrote, torch overwrites the first sources behind them.  All values are small integers."""
    n = 4
    stream = torch.cuda.Stream() if side_stream else torch.cuda.current_stream()
    new = lambda c: [torch.zeros(c, dtype=torch.float32, device="cuda") for _ in range(n)]
    x, a, b, c, d, e, f = new(count), new(count), new(count), new(count), new(count), new(count // n), new(count // n * n)
    kw = dict(dtype=nb.NUNA_F32)
    nb.nuna_init(4 * count + 16)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for it in range(1, 25):
            for r in range(n):
                x[r].fill_(it % 5 + r)
            nb.nuna_allreduce_oneshot(x, a, count, **kw)
            for r in range(n):
                x[r].fill_(-1000.0)
            nb.nuna_allreduce_twoshot(a, b, count, **kw)
            nb.nuna_allreduce_twoshot(b, c, count, flags=nb.NUNA_TWOSHOT_PUT, **kw)
            nb.nuna_alltoall(c, d, count // n, **kw)
            nb.nuna_reduce_scatter(d, e, count // n, **kw)
            nb.nuna_allgather(e, f, count // n, **kw)
            want = float((4 * (it % 5) + 6) * n * n * n)
            out = [t.clone() for t in f]
            for t in f:
                t.zero_()
            if it % 6 == 0:
                assert all(bool((t == want).all()) for t in out)
    assert nb.nuna_device_status() == nb.NUNA_OK


FORMS = {"co-located": nb.NUNA_PLACE_AWARE, "staged": nb.NUNA_PLACE_AWARE | nb.NUNA_PLACE_STAGED,
         "cluster": nb.NUNA_PLACE_AWARE | nb.NUNA_PLACE_CLUSTER, "lists": nb.NUNA_PLACE_AWARE | nb.NUNA_PLACE_SM_LISTS,
         "registers": nb.NUNA_PLACE_AWARE | nb.NUNA_PLACE_REGS, "auto": nb.NUNA_PLACE_AUTO,
         "resident": nb.NUNA_PLACE_AUTO | nb.NUNA_HINT_RESIDENT}


@pytest.mark.parametrize("shard", [3, 701, 17501])
@pytest.mark.parametrize("form", FORMS)
def test_every_one_shot_form_and_the_ragged_kernels_keep_stream_order(form, shard):
    """As above through the other forms of the one-shot, the allocation-free two-shot and, with shards that are no whole
    number of vectors, the ragged kernels: each call reads what the one before wrote, and has its sources overwritten."""
    n, count = 4, 4 * shard
    new = lambda c: [torch.zeros(c, dtype=torch.float32, device="cuda") for _ in range(n)]
    x, a, b, c, d, e, f = new(count), new(count), new(count), new(count), new(count), new(shard), new(count)
    kw = dict(dtype=nb.NUNA_F32)
    nb.nuna_allreduce_oneshot(x, a, count, flags=FORMS[form], **kw)            # builds what a form keeps per shape
    torch.cuda.synchronize()
    for it in range(1, 25):
        for r in range(n):
            x[r].fill_(it % 5 + r)
        nb.nuna_allreduce_oneshot(x, a, count, flags=FORMS[form], **kw)
        for r in range(n):
            x[r].fill_(-1000.0)
        nb.nuna_allreduce_oneshot(a, b, count, flags=FORMS[form], **kw)
        for r in range(n):
            a[r].fill_(-2000.0)
        nb.nuna_allreduce_twoshot_static(b, c, count, **kw)
        nb.nuna_alltoall(c, d, shard, **kw)
        nb.nuna_reduce_scatter(d, e, shard, **kw)
        nb.nuna_allgather(e, f, shard, **kw)
        for r in range(n):
            e[r].fill_(-3000.0)
        want = float((4 * (it % 5) + 6) * n * n * n)
        out = [t.clone() for t in f]
        for t in f:
            t.zero_()
        if it % 6 == 0:
            assert all(bool((t == want).all()) for t in out), it
    assert nb.nuna_device_status() == nb.NUNA_OK
