"""Which host buffers the host-buffer entry point works on in place, and with what result."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2608_00867_b200 import binding as nb

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
