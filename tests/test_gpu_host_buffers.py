"""Which host buffers the host-buffer entry point works on in place, and with what result."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2608_00867_b200 import binding as nb
from paper_2608_00867_b200 import workloads

pytestmark = pytest.mark.gpu

PAGE = 4096


def mapped(at, nbytes):
    f = nb.lib().nuna_debug_host_mapped
    f.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
    return f(at, nbytes)


def test_a_buffer_is_mapped_only_if_all_of_it_is_page_locked():
    rt = torch.cuda.cudart()
    torch.cuda.current_stream()
    room = np.zeros(9 * PAGE, dtype=np.uint8)
    a = (room.ctypes.data + PAGE - 1) // PAGE * PAGE
    assert mapped(a, 16) == 0
    assert int(rt.cudaHostRegister(a, 2 * PAGE, 0)) == 0
    try:
        assert mapped(a, 2 * PAGE) == 1 and mapped(a + 16, 2 * PAGE - 16) == 1 and mapped(a + 2 * PAGE - 16, 16) == 1
        assert mapped(a, 2 * PAGE + 1) == 0 and mapped(a + 16, 4 * PAGE) == 0      # the end is not
        assert int(rt.cudaHostRegister(a + 3 * PAGE, PAGE, 0)) == 0
        assert mapped(a, 4 * PAGE) == 0                                            # a page in the middle is not
        assert int(rt.cudaHostUnregister(a + 3 * PAGE)) == 0
        assert int(rt.cudaHostRegister(a + 2 * PAGE, 2 * PAGE, 0)) == 0
        assert mapped(a, 4 * PAGE) == 1 and mapped(a + PAGE, 2 * PAGE) == 1        # registered in two parts
        assert int(rt.cudaHostUnregister(a + 2 * PAGE)) == 0
    finally:
        rt.cudaHostUnregister(a)
    assert mapped(a, 16) == 0
    t = torch.zeros(3 << 20, dtype=torch.uint8).pin_memory()
    assert mapped(t.data_ptr(), 3 << 20) == 1 and mapped(t.data_ptr() + 16, (3 << 20) - 16) == 1
    assert mapped(torch.zeros(64, device="cuda").data_ptr(), 16) == 0


WORD = {"bf16": np.uint16, "f16": np.uint16, "f32": np.uint32}
GUARD = 64


@pytest.mark.parametrize("flags", [0, nb.NUNA_PLACE_AUTO, nb.NUNA_HINT_RESIDENT, nb.NUNA_PLACE_AWARE, nb.NUNA_PLACE_AUTO | nb.NUNA_LAUNCH_PDL])
@pytest.mark.parametrize("dtype", ["bf16", "f16", "f32"])
def test_one_shot_on_page_locked_buffers(dtype, flags):
    """In place (but for NUNA_PLACE_AWARE, which stages): ragged counts, several passes of the few blocks, buffers that are
    page-locked but not aligned to a vector, guard zones around the destinations."""
    word = WORD[dtype]
    size = np.dtype(word).itemsize
    for n, count in ((2, 5), (8, 1001), (3, 40 * 2048 + 3), (16, 4096)):
        src = workloads.rank_buffers_typed(n, count, "normal", 11 + count, dtype)
        want = oracle.allreduce(src, dtype=dtype)[0]
        for shift in (0, size):
            psrc, pdst = [], []
            for a in src:
                t = torch.zeros(shift + a.nbytes, dtype=torch.uint8)
                t[shift:] = torch.from_numpy(a.view(np.uint8).copy())
                psrc.append(t.pin_memory())
                pdst.append(torch.full((a.nbytes + 2 * GUARD + shift,), 0x5A, dtype=torch.uint8).pin_memory())
            nb.nuna_allreduce_host([t.data_ptr() + shift for t in psrc], [t.data_ptr() + GUARD + shift for t in pdst], count,
                                   dtype=nb.DTYPE_BY_NAME[dtype], flags=flags)
            for t in pdst:
                h = t.numpy()
                at = GUARD + shift
                assert (h[:at] == 0x5A).all() and (h[at + want.nbytes:] == 0x5A).all(), (n, count, shift)
                assert np.array_equal(h[at:at + want.nbytes].view(word), want), (n, count, shift)
    assert nb.nuna_device_status() == nb.NUNA_OK
