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
