"""Calls in a captured graph without NUNA_LAUNCH_PDL: what they choose there (nuna_allreduce's plain crossovers, the tiles
without a prefetch) is reached by no eager call.  And the eager crossovers of few ranks.  Bit for bit against a rank-ordered
binary32 fold in torch."""
import pytest
import torch

from paper_2608_00867_b200 import binding as nb

pytestmark = pytest.mark.gpu

KIB, MIB = 1 << 10, 1 << 20
GUARD = 64
# the largest message, in bytes per rank, that the one-shot takes when launched plainly; with NUNA_TWOSHOT_SYNC; and the
# messages around which NUNA_PLACE_AUTO changes its one-shot kernel, or leaves it
PLAIN = {2: 1 * MIB, 4: 512 * KIB, 8: 64 * KIB, 16: 8 * KIB}
SYNC = {2: 8 * MIB, 4: 4 * MIB, 8: 1 * MIB, 16: 512 * KIB}
AUTO = {2: [1 * MIB], 4: [512 * KIB], 8: [128 * KIB], 16: [64 * KIB, 1 * MIB]}
AUTO_SYNC = {2: [8 * MIB], 4: [4 * MIB], 8: [2 * MIB], 16: [512 * KIB]}


def make(n, elems, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return [torch.randn(elems, generator=gen, device="cuda").bfloat16() for _ in range(n)]


def fold(parts):
    acc = parts[0].float()
    for s in parts[1:]:
        acc = acc + s.float()
    return acc.bfloat16()


def captured(call, *args, **kw):
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        call(*args, **kw)
    g.replay()
    g.replay()
    torch.cuda.synchronize()


def guarded(n, elems):
    return [torch.full((elems + GUARD,), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(n)]


def check(dst, want, what):
    for d, w in zip(dst, want):
        assert torch.equal(d[:w.numel()], w), what
        assert bool((d[w.numel():] == 7.0).all()), (what, "written beyond the end")


def allreduce(n, sizes, flags, graph, seed):
    top = max(sizes) // 2 + 16
    src = make(n, top, seed)
    whole = fold(src)
    nb.nuna_init(2 * top)
    for size in sizes:
        for vectors in (-1, 0, 1):
            count = size // 2 + 8 * vectors + (3 if vectors > 0 else 0)
            dst = guarded(n, count)
            (captured if graph else lambda f, *a, **k: f(*a, **k))(nb.nuna_allreduce, src, dst, count, flags=flags)
            check(dst, [whole[:count]] * n, (n, count, flags, graph))
    assert nb.nuna_device_status() == nb.NUNA_OK


@pytest.mark.parametrize("n", [2, 4, 8, 16])
def test_captured_allreduce_on_both_sides_of_the_plain_crossovers(n):
    allreduce(n, [PLAIN[n]], 0, True, n)
    allreduce(n, [PLAIN[n]], nb.NUNA_HINT_RESIDENT, True, n)
    allreduce(n, [SYNC[n]], nb.NUNA_TWOSHOT_SYNC, True, n + 1)
    allreduce(n, AUTO[n], nb.NUNA_PLACE_AUTO, True, n + 2)
    allreduce(n, AUTO_SYNC[n], nb.NUNA_PLACE_AUTO | nb.NUNA_TWOSHOT_SYNC, True, n + 3)


@pytest.mark.parametrize("n", [2, 3, 4, 5, 16])
def test_eager_allreduce_on_both_sides_of_its_crossovers(n):
    allreduce(n, [16 * KIB, 256 * KIB], 0, False, n)
    allreduce(n, [16 * KIB, 256 * KIB], nb.NUNA_HINT_RESIDENT, False, n)
    allreduce(n, [MIB], nb.NUNA_PLACE_AUTO, False, n)
    allreduce(n, [SYNC.get(n, MIB)], nb.NUNA_TWOSHOT_SYNC, False, n)


@pytest.mark.parametrize("shard", [8, 4096, 30011, 131072])
@pytest.mark.parametrize("n", [2, 5, 8, 16])
def test_captured_collectives_without_dependent_launch(n, shard):
    big = make(n, n * shard, 3 * n + shard)
    small = [b[:shard].clone() for b in big]
    total = fold(big)
    dst = guarded(n, shard)
    captured(nb.nuna_reduce_scatter, big, dst, shard)
    check(dst, [total[r * shard:(r + 1) * shard] for r in range(n)], "reduce-scatter")
    dst = guarded(n, n * shard)
    captured(nb.nuna_allgather, small, dst, shard)
    check(dst, [torch.cat(small)] * n, "allgather")
    dst = guarded(n, n * shard)
    captured(nb.nuna_alltoall, big, dst, shard)
    check(dst, [torch.cat([big[r][d * shard:(d + 1) * shard] for r in range(n)]) for d in range(n)], "alltoall")
    for flags in (nb.NUNA_PLACE_AWARE | nb.NUNA_PLACE_REGS, nb.NUNA_PLACE_AWARE | nb.NUNA_PLACE_REGS | nb.NUNA_HINT_RESIDENT):
        dst = guarded(n, n * shard)
        captured(nb.nuna_allreduce_oneshot, big, dst, n * shard, flags=flags)
        check(dst, [total] * n, ("registers", flags))
    dst = guarded(n, n * shard)
    captured(nb.nuna_allreduce_twoshot, big, dst, n * shard, flags=nb.NUNA_TWOSHOT_PUT)
    check(dst, [total] * n, "put")
    assert nb.nuna_device_status() == nb.NUNA_OK
