"""The register-sharing one-shot, the put form and the size-selected allreduce on both sides of every line of the rule
that chooses their tiles and blocks: vectors per SM (32, 56, 128, 448) and bytes of sources in total (6, 8, 16, 64 MiB),
one vector below, at and above it, with a ragged end.  Bit for bit against a rank-ordered binary32 fold in torch."""
import pytest
import torch

from paper_2608_00867_b200 import binding as nb

pytestmark = pytest.mark.gpu

SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148
GUARD = 64
CALLS = {"regs": (nb.nuna_allreduce_oneshot, nb.NUNA_PLACE_AWARE | nb.NUNA_PLACE_REGS),
         "put": (nb.nuna_allreduce_twoshot, nb.NUNA_TWOSHOT_PUT),
         "auto": (nb.nuna_allreduce, nb.NUNA_PLACE_AUTO), "plain": (nb.nuna_allreduce, 0)}


def vectors(n):
    per_sm = [SMS * u for u in (1, 16, 32, 56, 64, 128, 448)]
    total = [(m << 20) // 16 // n for m in (6, 8, 16, 64)]
    return sorted({v + d for v in per_sm + total for d in (-1, 0, 1)})


@pytest.mark.parametrize("n,dtype", [(2, "bf16"), (3, "f32"), (4, "f16"), (8, "bf16"), (8, "f32"), (12, "bf16"), (16, "f16")])
def test_both_sides_of_every_line(n, dtype):
    tdt, code = {"bf16": (torch.bfloat16, 0), "f16": (torch.float16, 1), "f32": (torch.float32, 2)}[dtype]
    per_vec = 16 // tdt.itemsize
    top = vectors(n)[-1] * per_vec + per_vec
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    src = [torch.randn(top, generator=gen, device="cuda").to(tdt) for _ in range(n)]
    acc = src[0].to(torch.float32, copy=True)
    for s in src[1:]:
        acc += s.float()
    want = acc.to(tdt)
    del acc
    dst = [torch.empty(top + GUARD, dtype=tdt, device="cuda") for _ in range(n)]
    for vec in vectors(n):
        count = vec * per_vec + (vec % per_vec)               # ragged for most
        small = vec < 64 * SMS
        for name, (call, flags) in CALLS.items():
            for more in ((0, nb.NUNA_HINT_RESIDENT) if small or name == "regs" else (0,)):
                for d in dst:
                    d[:count + GUARD].fill_(7.0)
                call(src, dst, count, dtype=code, flags=flags | more | nb.NUNA_LAUNCH_PDL)
                for d in dst:
                    assert torch.equal(d[:count], want[:count]), (name, more, count)
                    assert bool((d[count:count + GUARD] == 7.0).all()), (name, more, count, "written beyond the end")
    assert nb.nuna_device_status() == nb.NUNA_OK
