"""Reduce-scatter, allgather and alltoall of shards that are no whole number of 16-byte vectors, at the edges of their
tiles (248 result vectors, 16 ... 224 vectors, 448 vectors): every phase of a shard against the vectors, no vector at
all, one vector, one element around a tile.  Bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_00867_b200 import binding as nb
from paper_2608_00867_b200 import workloads

pytestmark = pytest.mark.gpu

GUARD = 64
WORD = {"bf16": np.uint16, "f16": np.uint16, "f32": np.uint32}
SHARDS = [1, 3, 7, 9, 15, 17, 23, 129, 248 * 8 - 1, 248 * 8 + 1, 256 * 8 + 3, 221 * 8 + 1, 217 * 8 + 7, 448 * 8 - 1, 448 * 8 + 9, 30011]


def upload(arrs):
    return [torch.from_numpy(a.view(np.uint8).copy()).cuda() for a in arrs]


def outputs(n, nbytes):
    full = [torch.full((nbytes + 2 * GUARD,), 0x5A, dtype=torch.uint8, device="cuda") for _ in range(n)]
    return full, [t.data_ptr() + GUARD for t in full]


def check(full, want, word):
    torch.cuda.synchronize()
    for t, w in zip(full, want):
        h = t.cpu().numpy()
        assert (h[:GUARD] == 0x5A).all() and (h[GUARD + w.nbytes:] == 0x5A).all(), "guard zone overwritten"
        assert np.array_equal(h[GUARD:GUARD + w.nbytes].view(word), w)


@pytest.mark.parametrize("shard", SHARDS)
@pytest.mark.parametrize("n", [2, 3, 8, 16])
@pytest.mark.parametrize("dtype", ["bf16", "f16", "f32"])
def test_ragged_shards(dtype, n, shard):
    word, code = WORD[dtype], nb.DTYPE_BY_NAME[dtype]
    size = np.dtype(word).itemsize
    big = workloads.rank_buffers_typed(n, n * shard, "normal", 5 + shard, dtype)
    small = [b[:shard].copy() for b in big]
    dbig, dsmall = upload(big), upload(small)
    for flags in (0, nb.NUNA_LAUNCH_PDL | nb.NUNA_HINT_RESIDENT):
        full, dst = outputs(n, shard * size)
        nb.nuna_reduce_scatter(dbig, dst, shard, dtype=code, flags=flags)
        check(full, oracle.reduce_scatter(big, dtype=dtype), word)
        full, dst = outputs(n, n * shard * size)
        nb.nuna_allgather(dsmall, dst, shard, dtype=code, flags=flags)
        check(full, [np.concatenate(small)] * n, word)
        full, dst = outputs(n, n * shard * size)
        nb.nuna_alltoall(dbig, dst, shard, dtype=code, flags=flags)
        check(full, [np.concatenate([big[r][d * shard:(d + 1) * shard] for r in range(n)]) for d in range(n)], word)
    assert nb.nuna_device_status() == nb.NUNA_OK
