"""The reduce-scatter that prefetches and releases its successor early: shards around the edges of its tiles of 128, 192 and
256 vectors and around the lines where it takes over and where its tile changes, against a rank-ordered binary32 fold in
torch; and replayed runs in which every call reads what the one before it wrote."""
import pytest
import torch

from paper_2608_00867_b200 import binding as nb

pytestmark = pytest.mark.gpu

SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148


@pytest.mark.parametrize("n", [2, 4, 5, 8, 9, 16])
def test_tiles_and_lines(n):
    first = ((64 if n <= 4 else 32) // n) * 256                     # vectors of a shard: below it the ordinary kernel runs
    wave = SMS * 4 * 256 // n // 256 * 256                          # the longest shard of one wave of full tiles
    vectors = [1, 127, 128, 129, 191, 192, 193, 255, 256, 257, first - 1, first, first + 1, wave, wave + 1, wave + 129]
    if n > 8:
        vectors += [(64 << 20) // 16 // n // n, (64 << 20) // 16 // n // n + 129]     # 64 MiB of sources: the tile is wide again beyond
    top = 8 * n * max(vectors)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    src = [torch.randn(top, generator=gen, device="cuda").bfloat16() for _ in range(n)]
    for shard in (8 * v for v in vectors if v > 0):
        acc = src[0][:n * shard].float()
        for s in src[1:]:
            acc = acc + s[:n * shard].float()
        want = acc.bfloat16()
        for flags in (0, nb.NUNA_LAUNCH_PDL, nb.NUNA_HINT_RESIDENT):
            dst = [torch.full((shard + 64,), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(n)]
            nb.nuna_reduce_scatter(src, dst, shard, flags=flags)
            for r, d in enumerate(dst):
                assert torch.equal(d[:shard], want[r * shard:(r + 1) * shard]) and bool((d[shard:] == 7.0).all()), (shard, flags)
    assert nb.nuna_device_status() == nb.NUNA_OK


@pytest.mark.parametrize("shard", [4096, 16384, 70000])
def test_replayed_runs_read_what_was_just_written(shard):
    """alltoall -> reduce-scatter -> allgather, four times over in one graph with dependent launches: a prefetch that came too
    early may fetch old data into L2, and must not be seen.  Small integers, so every sum is exact."""
    n = 8
    new = lambda c: [torch.zeros(c, dtype=torch.float32, device="cuda") for _ in range(n)]
    a, b, c = new(n * shard), new(n * shard), new(shard)
    kw = dict(dtype=nb.NUNA_F32, flags=nb.NUNA_LAUNCH_PDL)
    nb.nuna_alltoall(a, b, shard, **kw)                             # the context exists
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        for _ in range(4):
            nb.nuna_alltoall(a, b, shard, **kw)
            nb.nuna_reduce_scatter(b, c, shard, **kw)
            nb.nuna_allgather(c, a, shard, **kw)
    for it in range(1, 7):
        for r in range(n):
            a[r].copy_(torch.arange(n * shard, device="cuda") % 7 + r + it)
        x = torch.stack(a)
        for _ in range(4):                                          # b[d] = concatenated blocks, c[r] = their sums, a[d] = all of c
            x = x.view(n, n, shard).transpose(0, 1).reshape(n, n * shard).sum(0).expand(n, n * shard)
        g.replay()
        torch.cuda.synchronize()
        for t in a:
            assert torch.equal(t, x[0]), it
