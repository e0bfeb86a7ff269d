"""The register-sharing one-shot and the put form with a block per tile and with a capped grid that loops over the tiles,
cold and L2-resident: no vector at all, a ragged end only, one vector around a tile, several tiles per block.  Bit for bit
against the oracle, with guard zones."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_00867_b200 import binding as nb
from paper_2608_00867_b200 import workloads

pytestmark = pytest.mark.gpu

GUARD = 64
FORMS = [(nb.nuna_allreduce_oneshot, nb.NUNA_PLACE_AWARE | nb.NUNA_PLACE_REGS), (nb.nuna_allreduce_twoshot, nb.NUNA_TWOSHOT_PUT)]


@pytest.mark.parametrize("blocks", [0, 1, 7])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("n", [1, 2, 4, 5, 8, 9, 16])
def test_block_per_tile_and_capped_grid(n, dtype, blocks):
    code, word = nb.DTYPE_BY_NAME[dtype], np.uint16 if dtype == "bf16" else np.uint32
    size = np.dtype(word).itemsize
    try:
        nb.nuna_set_option(nb.NUNA_OPT_BLOCKS, blocks)
        for vectors in (0, 1, 15, 16, 17, 63, 65, 500):
            for ragged in (0, 16 // size - 1):
                count = vectors * (16 // size) + ragged
                if count == 0:
                    continue
                src = workloads.rank_buffers_typed(n, count, "normal", 3 + count, dtype)
                want = oracle.allreduce(src, dtype=dtype)[0]
                dsrc = [torch.from_numpy(a.view(np.uint8).copy()).cuda() for a in src]
                for call, flags in FORMS:
                    for more in (0, nb.NUNA_HINT_RESIDENT):
                        full = [torch.full((count * size + 2 * GUARD,), 0x5A, dtype=torch.uint8, device="cuda") for _ in range(n)]
                        call(dsrc, [t.data_ptr() + GUARD for t in full], count, dtype=code, flags=flags | more)
                        for t in full:
                            h = t.cpu().numpy()
                            assert (h[:GUARD] == 0x5A).all() and (h[GUARD + count * size:] == 0x5A).all(), (count, flags, more)
                            assert np.array_equal(h[GUARD:GUARD + count * size].view(word), want), (count, flags, more)
    finally:
        nb.nuna_set_option(nb.NUNA_OPT_BLOCKS, 0)
    assert nb.nuna_device_status() == nb.NUNA_OK


SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148
L2 = torch.cuda.get_device_properties(0).L2_cache_size if torch.cuda.is_available() else 126 << 20


@pytest.mark.parametrize("n", [2, 5, 7, 9, 16])
def test_resident_shapes_on_both_sides_of_every_line(n):
    """Vectors per SM (32, 64, 128, 256, 384, 448, 1000) and a quarter of L2 in sources, one vector below, at and above."""
    lines = [SMS * u for u in (32, 64, 128, 256, 384, 448, 1000)] + [L2 // 4 // 16 // n]
    top = 8 * (max(lines) + 2)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    src = [torch.randn(top, generator=gen, device="cuda").bfloat16() for _ in range(n)]
    acc = src[0].float()
    for s in src[1:]:
        acc += s.float()
    want = acc.bfloat16()
    dst = [torch.empty(top + GUARD, dtype=torch.bfloat16, device="cuda") for _ in range(n)]
    for vectors in sorted({v + d for v in lines for d in (-1, 0, 1)}):
        count = 8 * vectors + vectors % 8
        for call, flags in FORMS:
            for d in dst:
                d[:count + GUARD].fill_(7.0)
            call(src, dst, count, flags=flags | nb.NUNA_HINT_RESIDENT)
            for d in dst:
                assert torch.equal(d[:count], want[:count]), (count, flags)
                assert bool((d[count:count + GUARD] == 7.0).all()), (count, flags)
    assert nb.nuna_device_status() == nb.NUNA_OK


@pytest.mark.parametrize("n", [3, 4, 7, 8, 16])
def test_allgather_on_both_sides_of_the_block_width_lines(n):
    """Tiles of 104 ... 184 vectors: blocks become as wide as their tiles at 112 (from 8 ranks) and 176 (from 4)."""
    for tile in (104, 112, 168, 176, 184):
        for vectors in (tile * 4 * SMS // n, tile * 4 * SMS // n // 8 * 8, tile * 4 * SMS // n - 3):
            src = [torch.randint(0, 1 << 15, (8 * vectors,), device="cuda", dtype=torch.int16) for _ in range(n)]
            dst = [torch.full((8 * vectors * n + GUARD,), -7, device="cuda", dtype=torch.int16) for _ in range(n)]
            nb.nuna_allgather(src, dst, 8 * vectors)
            want = torch.cat(src)
            for d in dst:
                assert torch.equal(d[:want.numel()], want) and bool((d[want.numel():] == -7).all()), (n, tile, vectors)
    assert nb.nuna_device_status() == nb.NUNA_OK
