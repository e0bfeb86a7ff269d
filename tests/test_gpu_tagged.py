"""The two-shot whose shard words carry their own flags, and the one whose shard is the owners' destinations: no vector at all, a ragged end only, one vector around a tile, the
message sizes at which its shape and its range change, mixed with the other two-shot forms that draw from the same ticket
word, replayed, and with a wait that runs out.  Bit for bit against the oracle or a rank-ordered binary32 fold in torch."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_00867_b200 import binding as nb
from paper_2608_00867_b200 import workloads

pytestmark = pytest.mark.gpu

GUARD = 64
SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148


@pytest.mark.parametrize("dtype", ["bf16", "f16", "f32"])
@pytest.mark.parametrize("n", [1, 2, 3, 8, 9, 16])
def test_small_and_ragged(n, dtype):
    code, word = nb.DTYPE_BY_NAME[dtype], np.uint16 if dtype != "f32" else np.uint32
    size = np.dtype(word).itemsize
    for vectors in (0, 1, 7, 8, 31, 32, 33, 64, 65, 500):
        for ragged in (0, 1, 16 // size - 1):
            count = vectors * (16 // size) + ragged
            if count == 0:
                continue
            src = workloads.rank_buffers_typed(n, count, "normal", 5 + count, dtype)
            src[0][: min(count, 3)] = np.array([0x7FFF, 0xFFFF, 0x7F80][: min(count, 3)] if size == 2 else
                                               [0x7FFFFFFF, 0xFFFFFFFF, 0x7F800000][: min(count, 3)], dtype=word)
            want = oracle.allreduce(src, dtype=dtype)[0]
            mag = {"bf16": (0x7FFF, 0x7F80), "f16": (0x7FFF, 0x7C00), "f32": (0x7FFFFFFF, 0x7F800000)}[dtype]
            nan = (want & word(mag[0])) > mag[1]
            dsrc = [torch.from_numpy(a.view(np.uint8).copy()).cuda() for a in src]
            full = [torch.full((count * size + 2 * GUARD,), 0x5A, dtype=torch.uint8, device="cuda") for _ in range(n)]
            nb.nuna_allreduce_twoshot(dsrc, [t.data_ptr() + GUARD for t in full], count, dtype=code)
            for t in full:
                h = t.cpu().numpy()
                assert (h[:GUARD] == 0x5A).all() and (h[GUARD + count * size:] == 0x5A).all(), count
                got = h[GUARD:GUARD + count * size].view(word)
                assert np.array_equal((got & word(mag[0])) > mag[1], nan) and np.array_equal(got[~nan], want[~nan]), count
    assert nb.nuna_device_status() == nb.NUNA_OK


@pytest.mark.parametrize("n", [2, 4, 8, 16])
def test_both_sides_of_every_line_and_every_neighbour(n):
    """Vectors per rank around the lines of the shape and the end of the range; tagged, flagged and put calls in turn on one
    stream, so that each draws its tickets, and writes its tags, behind the others."""
    lines = [SMS * u for u in (8, 32, 96, 192, 224, 384, 512, 768)] + [((5 if n <= 2 else 6 if n <= 4 else 8) << 20) // 16]   # the last: end of the range
    top = 8 * (max(lines) + 2)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    src = [torch.randn(top, generator=gen, device="cuda").bfloat16() for _ in range(n)]
    acc = src[0].float()
    for s in src[1:]:
        acc = acc + s.float()
    want = acc.bfloat16()
    dst = [torch.zeros(top, dtype=torch.bfloat16, device="cuda") for _ in range(n)]
    for line in lines:
        for vectors in (line - 1, line, line + 1):
            count = 8 * vectors + 5
            for flags in (0, nb.NUNA_TWOSHOT_SYS_SCOPE, 0, nb.NUNA_TWOSHOT_PUT, nb.NUNA_LAUNCH_PDL | nb.NUNA_HINT_RESIDENT):
                for d in dst:
                    d.fill_(7.0)
                nb.nuna_allreduce_twoshot(src, dst, count, flags=flags)
                for d in dst:
                    assert torch.equal(d[:count], want[:count]) and bool((d[count:count + GUARD] == 7.0).all()), (count, flags)
    assert nb.nuna_device_status() == nb.NUNA_OK


TORCH = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}


def same(got, want):
    """Equal, NaN where there is to be one."""
    return bool(((got == want) | (torch.isnan(got) & torch.isnan(want))).all())


def fold(parts):
    """The sum in rank order in binary32, rounded once."""
    acc = parts[0].float()
    for s in parts[1:]:
        acc = acc + s.float()
    return acc.to(parts[0].dtype)


@pytest.mark.parametrize("dtype", TORCH)
@pytest.mark.parametrize("n,mib", [(1, 9), (2, 6), (2, 12), (2, 17), (3, 7), (3, 60), (4, 41), (5, 9), (6, 9), (7, 19), (8, 9), (8, 17)])
def test_shard_in_the_owners_destinations(n, mib, dtype):
    """Beyond the tagged form, on both sides of the lines where the shard moves into the destinations and its tile changes:
    counts that end in a whole tile, in the middle of one and in the middle of a vector; eager, captured plainly, with
    dependent launches and with the resident hint; infinities and NaN among the values."""
    size = nb.ELEM_SIZE[nb.DTYPE_BY_NAME[dtype]]
    top, vec = (mib << 20) // size, 16 // size
    gen = torch.Generator(device="cuda")
    gen.manual_seed(mib)
    src = [torch.randn(top, generator=gen, device="cuda").to(TORCH[dtype]) for _ in range(n)]
    src[0][7], src[n - 1][11], src[0][top // 2], src[n - 1][top // 2] = float("inf"), float("nan"), float("inf"), float("-inf")
    want = fold(src)
    nb.nuna_init(size * top)
    dst = [torch.zeros(top, dtype=TORCH[dtype], device="cuda") for _ in range(n)]
    for count in (top, top - vec * 4096, top - vec * 1001, top - vec * 333 - 3):
        for flags in (0, nb.NUNA_LAUNCH_PDL, nb.NUNA_LAUNCH_PDL | nb.NUNA_HINT_RESIDENT):
            call = lambda: nb.nuna_allreduce_twoshot(src, dst, count, dtype=nb.DTYPE_BY_NAME[dtype], flags=flags)
            g = torch.cuda.CUDAGraph()
            torch.cuda.synchronize()
            with torch.cuda.graph(g):
                call()
            for run in (call, g.replay):
                for d in dst:
                    d.fill_(7.0)
                run()
                run()
                for d in dst:
                    assert same(d[:count], want[:count]) and bool((d[count:] == 7.0).all()), (count, flags)
    assert nb.nuna_device_status() == nb.NUNA_OK


@pytest.mark.parametrize("form", ["tagged", "flags", "in place"])
@pytest.mark.parametrize("n,dtype", [(2, "bf16"), (2, "f16"), (4, "f32"), (6, "f32"), (8, "bf16"), (8, "f16"), (8, "f32")])
def test_every_call_reads_what_the_one_before_wrote(n, dtype, form):
    """Four calls in a row, eager and captured with dependent launches, whose prefetch goes out while the call before still
    writes what they read.  Whole numbers that differ from place to place and fit the type, infinities and NaN."""
    code = nb.DTYPE_BY_NAME[dtype]
    size = nb.ELEM_SIZE[code]
    count = {"tagged": 300 << 10, "flags": 300 << 10, "in place": (9 << 20) + (64 << 10)}[form] // size - 3
    flags = nb.NUNA_LAUNCH_PDL | (nb.NUNA_TWOSHOT_SYS_SCOPE if form == "flags" else 0)
    nb.nuna_init(size * count + 16)
    new = lambda: [torch.zeros(count, dtype=TORCH[dtype], device="cuda") for _ in range(n)]
    x, a, b = new(), new(), new()

    def run():
        for s, d in ((x, a), (a, b), (b, a), (a, b)):
            nb.nuna_allreduce_twoshot(s, d, count, dtype=code, flags=flags)

    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        run()
    place = torch.arange(count, device="cuda")
    for it in range(8):
        for r in range(n):
            x[r].copy_((place * (3 + it) % 31) // 4 + r % 2)
        x[0][5::4099], x[n - 1][7::4099], x[0][9::4099], x[n - 1][9::4099] = float("inf"), float("nan"), float("inf"), float("-inf")
        want = x
        for _ in range(4):
            want = [fold(want)] * n
        g.replay() if it % 2 else run()
        for t in b:
            assert same(t, want[0]), it
    assert nb.nuna_device_status() == nb.NUNA_OK


@pytest.mark.parametrize("pdl", [0, nb.NUNA_LAUNCH_PDL])
def test_back_to_back_replays_of_mixed_sizes(pdl):
    """A captured run in which every call reads what the one before wrote, sizes alternating, replayed and mixed with eager
    calls: a ticket drawn ahead of the wait must find the word set up by the launch before.  Every element of both buffers
    after every run; whole numbers below 2^24 that differ from place to place."""
    n, sizes = 4, (64, 70001, 8, 300000, 2049, 262144)
    top = max(sizes)
    nb.nuna_init(4 * top + 16)
    bufs = torch.zeros(2, n, top, device="cuda")
    ranks = [list(b) for b in bufs]

    def run():
        for k, c in enumerate(sizes):
            nb.nuna_allreduce_twoshot(ranks[k % 2], ranks[1 - k % 2], c, dtype=nb.NUNA_F32, flags=pdl)

    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        run()
    place = torch.arange(top, device="cuda")
    for it in range(20):
        bufs[0] = torch.stack([place * (2 + it) % 13 + r for r in range(n)])
        bufs[1].zero_()
        start = bufs.clone()
        for _ in range(1 + it % 3):
            bufs.copy_(start)
            g.replay() if it % 2 else run()
        want = start
        for k, c in enumerate(sizes):
            want[1 - k % 2, :, :c] = want[k % 2, :, :c].sum(0)
        assert torch.equal(bufs, want), it
    assert nb.nuna_device_status() == nb.NUNA_OK


def test_wait_for_a_tag_times_out_cleanly():
    """Consumers that wait for tags nobody writes: every wait runs out after 50 ms, the status word latches the timeout, and
    the next ordinary calls work."""
    w = workloads.config_decode_activation()
    src = workloads.make(w)
    want = oracle.allreduce(src, nthreads=4)[0]
    dsrc = [torch.from_numpy(a.view(np.int16).copy()).cuda() for a in src]
    dst = [torch.zeros(w.count, dtype=torch.int16, device="cuda") for _ in range(w.nranks)]
    assert nb.debug_twoshot(dsrc, dst, w.count, timeout_ms=50, unset_flags=True, tagged=True) == nb.NUNA_OK
    torch.cuda.synchronize()
    assert all(not bool(d.any()) for d in dst)
    assert nb.nuna_device_status() == nb.NUNA_ERR_TIMEOUT
    assert nb.nuna_device_status() == nb.NUNA_OK
    for _ in range(2):
        nb.nuna_allreduce_twoshot(dsrc, dst, w.count)
        for d in dst:
            assert np.array_equal(d.cpu().numpy().view(np.uint16), want)
    assert nb.nuna_device_status() == nb.NUNA_OK


def test_growing_messages_leave_little_behind():
    """Outgrown scratch stays allocated for the graphs that may name it.  Messages that grow to 8 MiB in steps of 512 KiB leave
    one shard per step behind, but not twice as much again in slots: 68 MiB of shards (in pages of 2 MiB) and 32 of slots."""
    mib = 1 << 20
    n, count = 2, 2 * mib
    src = [torch.full((count,), float(r + 1), dtype=torch.bfloat16, device="cuda") for r in range(n)]
    dst = [torch.zeros_like(s) for s in src]
    nb.lib().nuna_shutdown()
    nb.nuna_init(4096)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for k in range(1, 17):
        nb.nuna_init(k * mib // 2)
    used = free - torch.cuda.mem_get_info()[0]
    assert used <= (68 + 16 * 2 + 32 + 8) * mib, used / mib
    nb.nuna_allreduce_twoshot(src, dst, count)                      # and what is there now is used: 4 MiB per rank, tagged
    nb.nuna_device_status()
    assert nb.lib().nuna_shutdown() == nb.NUNA_OK
    assert torch.cuda.mem_get_info()[0] >= free - 16 * mib          # all of it is given back, but for kernels loaded since
    assert all(bool((d == 3.0).all()) for d in dst) and nb.nuna_device_status() == nb.NUNA_OK
