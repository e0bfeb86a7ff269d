"""Which kernel a call runs, read from a trace, on both sides of the lines that a rule draws between two of them."""
import warnings

import pytest
import torch

from paper_2608_00867_b200 import binding as nb

pytestmark = pytest.mark.gpu

MIB = 1 << 20


def kernels(call):
    """Names of the kernels that the call launches, without their template arguments but for one that is a truth value."""
    call()
    torch.cuda.synchronize()
    with warnings.catch_warnings():
        warnings.simplefilter("ignore")
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as trace:
            call()
            torch.cuda.synchronize()
    names = [e.key for e in trace.key_averages() if "nuna::" in e.key]
    if not names:
        pytest.skip("nothing can be traced here")
    return {name.split("nuna::")[1].split("<")[0].split("(")[0] + (" true" if "true>" in name else "") for name in names}


def reduce_scatter(n, nbytes, flags):
    count = nbytes // 2 // n // 8 * 8
    src = [torch.ones(n * count, dtype=torch.bfloat16, device="cuda") for _ in range(n)]
    dst = [torch.zeros(count, dtype=torch.bfloat16, device="cuda") for _ in range(n)]
    return kernels(lambda: nb.nuna_reduce_scatter(src, dst, count, flags=flags))


@pytest.mark.parametrize("n,line_mib", [(2, 32), (8, 32), (16, 48)])
def test_reduce_scatter_runs_ahead_unasked_only_where_no_predecessor_makes_it_slower(n, line_mib):
    """`line_mib`: MiB of sources from which it does.  With NUNA_LAUNCH_PDL it also does below."""
    ahead, ordinary = {"k_reduce_scatter_ahead"}, {"k_reduce_scatter"}
    line = line_mib * MIB // n
    assert reduce_scatter(n, line, 0) == ahead
    assert reduce_scatter(n, line - 16 * n, 0) == ordinary
    assert reduce_scatter(n, line - 16 * n, nb.NUNA_LAUNCH_PDL) == ahead
    assert reduce_scatter(n, line, nb.NUNA_HINT_RESIDENT) == ordinary


def twoshot(n, nbytes, flags):
    count = nbytes // 2
    src = [torch.ones(count, dtype=torch.bfloat16, device="cuda") for _ in range(n)]
    dst = [torch.zeros(count, dtype=torch.bfloat16, device="cuda") for _ in range(n)]
    nb.nuna_init(nbytes)
    return kernels(lambda: nb.nuna_allreduce_twoshot(src, dst, count, flags=flags))


@pytest.mark.parametrize("n,cold,resident", [(2, 5, 5), (3, 6, 5), (4, 6, 5), (8, 8, 8)])
def test_the_largest_message_of_the_tagged_twoshot(n, cold, resident):
    """In MiB per rank, without and with the resident hint."""
    for flags, most in ((0, cold * MIB), (nb.NUNA_HINT_RESIDENT, resident * MIB)):
        assert twoshot(n, most, flags) == {"k_twoshot_tagged"}
        assert "k_twoshot_tagged" not in twoshot(n, most + 16, flags)


@pytest.mark.parametrize("n,mib,cold,resident", [(1, 9, True, True), (2, 10, True, True), (2, 16, True, False), (2, 17, True, True), (4, 16, True, True), (6, 16, True, True),
                                                 (7, 12, True, False), (8, 12, True, False), (8, 17, False, False)])
def test_the_flag_twoshot_reduces_in_place_where_that_pays(n, mib, cold, resident):
    """MiB per rank; the kernel's last template argument says whether the shard is the owners' destinations."""
    for flags, in_place in ((0, cold), (nb.NUNA_HINT_RESIDENT, resident)):
        assert twoshot(n, mib * MIB, flags) == {"k_twoshot_flags" + (" true" if in_place else "")}
