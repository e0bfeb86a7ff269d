"""Argument marshalling of the native half of the binding: every form a rank buffer, a stream or a number may take.
No GPU: the library's own argument checks tell what arrived (they run before any CUDA call)."""
import os
import subprocess
import sys
import weakref

import numpy as np
import pytest
import torch

from paper_2608_00867_b200 import binding as nb
from paper_2608_00867_b200 import build as nbuild

A = 1 << 20                                  # fake aligned addresses; validation never dereferences them


@pytest.fixture(scope="module", autouse=True)
def built_library():
    nbuild.build()


class Buf:
    def __init__(self, addr):
        self.addr = addr

    def data_ptr(self):
        return self.addr


class Sub(torch.Tensor):
    pass


@pytest.mark.parametrize("n", [1, 2, 16, 17, 40])
@pytest.mark.parametrize("wrap", [list, tuple, iter])
def test_table_forms(n, wrap):
    src, dst = [A + 64 * i for i in range(n)], [Buf(2 * A + 64 * i) for i in range(n)]
    want = nb.NUNA_ERR_TOO_MANY_RANKS if n > 16 else nb.NUNA_ERR_TOO_LARGE
    assert nb.nuna_allreduce(wrap(src), wrap(dst), (1 << 40) + 1, stream=0, check=False) == want
    dst[-1] = Buf(2 * A + 64 * (n - 1) + 2)
    if n <= 16:                              # the last entry arrived: it is the misaligned one
        assert nb.nuna_allreduce(wrap(src), wrap(dst), 8, stream=0, check=False) == nb.NUNA_ERR_ALIGNMENT


def test_buffers_of_an_iterator_live_until_the_call_is_made():
    alive = []

    class Watched(Buf):
        def __init__(self, addr):
            super().__init__(addr)
            alive.append(weakref.ref(self))

    class Last(Buf):                         # the last address that is read before the call
        def data_ptr(self):
            self.seen = [w() is not None for w in alive]
            return self.addr

    last = Last(2 * A + 64)
    status = nb.nuna_allreduce((Watched(A + 64 * i) for i in range(2)), [2 * A, last], 8, dtype=9, stream=0, check=False)
    assert status == nb.NUNA_ERR_UNSUPPORTED_DTYPE and last.seen == [True, True]


@pytest.mark.parametrize("kind", [torch.Tensor, torch.nn.Parameter, Sub])
def test_tensor_addresses_are_the_tensors_own(kind):
    x = torch.zeros(64, dtype=torch.float32)
    x = torch.nn.Parameter(x) if kind is torch.nn.Parameter else x.as_subclass(Sub) if kind is Sub else x
    at = x.data_ptr()
    # alias with an address inside the tensor, none just behind it
    assert nb.nuna_allreduce([at + 16], [x], 8, dtype=nb.NUNA_F32, stream=0, check=False) == nb.NUNA_ERR_ALIAS
    assert nb.nuna_allreduce([at + 256 + 2], [x], 8, dtype=nb.NUNA_F32, stream=0, check=False) == nb.NUNA_ERR_ALIGNMENT
    y = np.zeros(64, dtype=np.float32)
    assert nb.nuna_allreduce_host([y], [int(y.ctypes.data) + 16], 8, dtype=nb.NUNA_F32, check=False) == nb.NUNA_ERR_ALIAS
    assert nb.nuna_allreduce_host([x], [at + 16], 8, dtype=nb.NUNA_F32, check=False) == nb.NUNA_ERR_ALIAS


def test_numbers_streams_and_errors():
    src, dst = [A, A + 4096], [A + 8192, A + 12288]

    class Stream:
        cuda_stream = 0

    assert nb.nuna_alltoall(src, dst, 0, stream=Stream()) == nb.NUNA_OK
    assert nb.nuna_alltoall(src, dst, np.int64(0), stream=0) == nb.NUNA_OK
    assert nb.nuna_allgather(src, dst, 8, stream=0, nranks=0, check=False) == nb.NUNA_ERR_INVALID_ARG
    assert nb.nuna_allgather(src, dst, 8, stream=0, nranks=3, check=False) == nb.NUNA_ERR_INVALID_ARG   # third rank: null
    assert nb.nuna_allreduce_twoshot_static(src, dst, 8, dtype=9, stream=0, check=False) == nb.NUNA_ERR_UNSUPPORTED_DTYPE
    with pytest.raises(nb.NunaError, match="nuna_reduce_scatter") as e:
        nb.nuna_reduce_scatter(src, src, 8, stream=0)
    assert e.value.status == nb.NUNA_ERR_ALIAS
    for bad in ((src, None, 8), (src, [None, None], 8), (src, dst, 1.5), (src, dst, "8")):
        with pytest.raises(TypeError):
            nb.nuna_allreduce(*bad, stream=0)


def test_arguments_by_name_and_position():
    """The native functions take their place on the first call and keep the names, the order and the defaults."""
    import inspect
    src, dst = [A, A + 4096], [A + 8192, A + 12288]
    for name, count in (("nuna_allreduce", "count"), ("nuna_reduce_scatter", "shard_count"), ("nuna_allgather", "shard_count"),
                        ("nuna_alltoall", "block_count")):
        call = getattr(nb, name)
        call(src, dst, 0, stream=0)
        native = getattr(nb, name)
        assert list(inspect.signature(native).parameters) == ["src", "dst", count, "dtype", "flags", "stream", "check", "nranks"]
        for f in (call, native):
            assert f(src, dst, 8, 9, 0, 0, False, 2) == nb.NUNA_ERR_UNSUPPORTED_DTYPE
            assert f(check=False, dst=dst, stream=0, src=src, dtype=9, **{count: 8}) == nb.NUNA_ERR_UNSUPPORTED_DTYPE
            assert f(src, dst, 8, nb.NUNA_BF16, 3, stream=0, check=False) == nb.NUNA_ERR_INVALID_ARG
            for args, kw in (((src, dst), {}), ((src, dst, 0), {"dst": dst}), ((src, dst, 0), {"nosuch": 1}), ((src,) * 9, {})):
                with pytest.raises(TypeError):
                    f(*args, **kw)


def test_a_module_built_for_another_torch_or_python_is_not_loaded(monkeypatch):
    import sysconfig
    assert torch.__version__ in os.path.basename(nbuild.native_path())
    assert nbuild.native_path().endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    monkeypatch.setattr(nbuild, "_torch_version", lambda: "0.0.1")
    monkeypatch.setattr(nb, "_native", None)
    with pytest.raises(RuntimeError, match="torch-0.0.1.*is missing"):
        nb._load_native()


def test_loading_the_native_module_keeps_what_the_caller_has_put_in_place():
    code = """
from paper_2608_00867_b200 import binding as nb
own = nb.nuna_allreduce
calls = []
def traced(*a, **k):
    calls.append(k["stream"])
    return own(*a, **k)
nb.nuna_allreduce = traced
other = nb.nuna_alltoall
src, dst = [1 << 20, (1 << 20) + 4096], [(1 << 20) + 8192, (1 << 20) + 12288]
assert nb.nuna_alltoall(src, dst, 0, stream=0) == 0                  # loads the native module
assert nb.nuna_alltoall is not other and nb.nuna_allreduce is traced
assert nb.nuna_allreduce(src, dst, 0, stream=0) == 0 and calls == [0]
"""
    run = subprocess.run([sys.executable, "-c", code], cwd=os.path.dirname(os.path.dirname(nb.__file__)), capture_output=True, text=True)
    assert run.returncode == 0, run.stderr
