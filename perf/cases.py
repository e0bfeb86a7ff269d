"""What a user of this library has it do, as cases that can be timed and compared.

A case is one call of a collective through ``paper_2608_00867_b200.binding`` (or one replay of a decode-step
chain), the way a tensor-parallel program issues it: rank buffers are torch tensors that exist before the call,
the call is asynchronous on the current stream, the results are the destination buffers.  Sizes are those of the
paper's inference traffic (Section 2.2: decode collectives are KB-range, prefill ones reach tens of MB) and of
the message-size sweep this repository benchmarks; ragged sizes stand for shapes that are no whole number of
16-byte vectors (odd vocabulary shards, odd token counts).
"""
from __future__ import annotations

import torch

from paper_2608_00867_b200 import binding as nb
from paper_2608_00867_b200 import workloads

KIB, MIB = 1 << 10, 1 << 20
DTYPES = {"bf16": (torch.bfloat16, nb.NUNA_BF16, 2), "f16": (torch.float16, nb.NUNA_F16, 2), "f32": (torch.float32, nb.NUNA_F32, 4)}
OPTIONS = {
    "default": 0,
    "pdl": nb.NUNA_LAUNCH_PDL,
    "auto": nb.NUNA_PLACE_AUTO,
    "auto_pdl": nb.NUNA_PLACE_AUTO | nb.NUNA_LAUNCH_PDL,
    # sources just written by a producing kernel, as a decode step's partial activations are
    "auto_pdl_resident": nb.NUNA_PLACE_AUTO | nb.NUNA_LAUNCH_PDL | nb.NUNA_HINT_RESIDENT,
    "put": nb.NUNA_TWOSHOT_PUT,
}
CHAIN_SETS = 2           # attention-out and MLP-out partials alternate


def listed():
    return [
        # the smallest call in use: two ranks, 8 KiB each; its latency is all that matters
        dict(name="allreduce_n2_8KiB", op="oneshot", n=2, count=4096, dtype="bf16", options="default"),
        # decode activation of eight-way tensor parallelism, batch 32 x hidden 8192, launched eagerly
        dict(name="allreduce_n8_512KiB", op="allreduce", n=8, count=32 * workloads.HIDDEN, dtype="bf16", options="auto_pdl"),
        # a mid-sized half-precision message with an odd element count and no options
        dict(name="allreduce_n4_ragged_f16", op="allreduce", n=4, count=1_000_003, dtype="f16", options="default"),
        # prefill: 4096 tokens x hidden 8192, the upper end of the size sweep
        dict(name="allreduce_n8_64MiB", op="allreduce", n=8, count=4096 * workloads.HIDDEN, dtype="bf16", options="auto_pdl"),
        # the flag-synchronised two-shot (the form that has a reduce-scatter and an allgather phase), 256 tokens
        dict(name="twoshot_n8_4MiB", op="twoshot", n=8, count=256 * workloads.HIDDEN, dtype="bf16", options="default"),
        # end to end from and to pinned host buffers
        dict(name="host_n8_512KiB", op="host", n=8, count=32 * workloads.HIDDEN, dtype="bf16", options="put"),
        # one decode step of an 80-layer model: 160 dependent allreduces, one token
        dict(name="chain_t1", op="chain", n=8, count=1 * workloads.HIDDEN, dtype="bf16", options="auto_pdl_resident"),
        # the same for a batch of 64 tokens
        dict(name="chain_t64", op="chain", n=8, count=64 * workloads.HIDDEN, dtype="bf16", options="auto_pdl_resident"),
        # sequence-parallel reduce-scatter of 4 MiB per rank
        dict(name="reduce_scatter_n8_4MiB", op="reduce_scatter", n=8, count=256 * KIB, dtype="bf16", options="pdl"),
        # reduce-scatter of an odd-sized binary32 gradient shard
        dict(name="reduce_scatter_n4_ragged_f32", op="reduce_scatter", n=4, count=262_147, dtype="f32", options="default"),
        # allgather of sixteen 64 KiB shards
        dict(name="allgather_n16_64KiB", op="allgather", n=16, count=32 * KIB, dtype="bf16", options="pdl"),
        # expert token routing: eight ranks, 64 KiB per (sender, receiver) pair
        dict(name="alltoall_n8_64KiB", op="alltoall", n=8, count=32 * KIB, dtype="bf16", options="pdl"),
    ]


def draw(rng):
    """`count` is elements per rank (allreduce forms), per shard (reduce-scatter, allgather) or per block (alltoall)."""
    def between(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    op = rng.choice(["oneshot", "allreduce", "allreduce", "twoshot", "host", "chain", "reduce_scatter", "allgather", "alltoall"])
    n = rng.choice([2, 3, 4, 6, 8, 8, 8, 12, 16])
    dtype = rng.choice(["bf16", "bf16", "f16", "f32"])
    size = DTYPES[dtype][2]
    options = rng.choice(["default", "pdl"])
    if op in ("oneshot", "allreduce"):
        options = rng.choice(["default", "auto", "auto_pdl", "auto_pdl", "auto_pdl_resident"])
        nbytes = between(8 * KIB, 512 * MIB // n)
    elif op == "twoshot":
        options = rng.choice(["default", "pdl", "put"])
        nbytes = between(8 * KIB, 512 * MIB // n)
    elif op == "host":
        options = rng.choice(["default", "put", "put"])
        nbytes = between(8 * KIB, 4 * MIB // n)
    elif op == "chain":
        n, dtype, options = 8, "bf16", rng.choice(["auto_pdl", "auto_pdl_resident"])
        count = between(1, 64) * workloads.HIDDEN
        return dict(op=op, n=n, count=count, dtype=dtype, options=options)
    else:
        nbytes = between(2 * KIB, 256 * MIB // (n * n))
    count = max(1, nbytes // size)
    if rng.random() < 0.5:                        # a whole number of 16-byte vectors; otherwise whatever came out, made odd
        count = (count + 7) // 8 * 8
    else:
        count |= 1
    return dict(op=op, n=n, count=count, dtype=dtype, options=options)


class _State:
    """Rank buffers and, for a chain, the handle that a program keeps for all its steps."""

    def __init__(self, case):
        self.op, self.n, self.count = case["op"], case["n"], case["count"]
        self.torch_dtype, self.dtype, _ = DTYPES[case["dtype"]]
        self.flags = OPTIONS[case["options"]]
        self.src, self.dst, self.chain = [], [], None

    def __del__(self):
        if self.chain is not None:
            nb.nuna_chain_destroy(self.chain)


def _sizes(case):
    """Elements of a source and of a destination buffer of one rank."""
    n, count = case["n"], case["count"]
    return {"reduce_scatter": (n * count, count), "allgather": (count, n * count),
            "alltoall": (n * count, n * count)}.get(case["op"], (count, count))


def prepare(case, seed):
    s = _State(case)
    src_elems, dst_elems = _sizes(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 1009 + 17)

    def values():                                 # N(0,1) activations, narrowed by torch
        return torch.randn(src_elems, generator=gen, device="cuda", dtype=torch.float32).to(s.torch_dtype)

    sets = CHAIN_SETS if s.op == "chain" else 1
    for _ in range(sets * s.n):
        if s.op == "host":
            s.src.append(values().cpu().pin_memory())
            s.dst.append(torch.zeros(dst_elems, dtype=s.torch_dtype).pin_memory())
        else:
            s.src.append(values())
            s.dst.append(torch.zeros(dst_elems, dtype=s.torch_dtype, device="cuda"))
    if s.op == "twoshot":
        nb.nuna_init(s.count * DTYPES[case["dtype"]][2] + 16)
    if s.op == "chain":
        split = [(s.src[k * s.n:(k + 1) * s.n], s.dst[k * s.n:(k + 1) * s.n]) for k in range(sets)]
        s.chain = nb.nuna_chain_create([a for a, _ in split], [b for _, b in split], workloads.CHAIN_NODES, s.count,
                                       dtype=s.dtype, flags=s.flags)
    return s


def run(s):
    if s.op == "oneshot":
        nb.nuna_allreduce_oneshot(s.src, s.dst, s.count, dtype=s.dtype, flags=s.flags)
    elif s.op == "allreduce":
        nb.nuna_allreduce(s.src, s.dst, s.count, dtype=s.dtype, flags=s.flags)
    elif s.op == "twoshot":
        nb.nuna_allreduce_twoshot(s.src, s.dst, s.count, dtype=s.dtype, flags=s.flags)
    elif s.op == "host":
        nb.nuna_allreduce_host(s.src, s.dst, s.count, dtype=s.dtype, flags=s.flags, two_shot=s.flags != 0)
    elif s.op == "chain":
        nb.nuna_chain_launch(s.chain)
    elif s.op == "reduce_scatter":
        nb.nuna_reduce_scatter(s.src, s.dst, s.count, dtype=s.dtype, flags=s.flags)
    elif s.op == "allgather":
        nb.nuna_allgather(s.src, s.dst, s.count, dtype=s.dtype, flags=s.flags)
    else:
        nb.nuna_alltoall(s.src, s.dst, s.count, dtype=s.dtype, flags=s.flags)
    return s.dst


def work(case):
    """Every source byte read once, every destination byte written once; one addition per element and further rank."""
    n, size = case["n"], DTYPES[case["dtype"]][2]
    src_elems, dst_elems = _sizes(case)
    nodes = workloads.CHAIN_NODES if case["op"] == "chain" else 1
    adds = 0 if case["op"] in ("allgather", "alltoall") else src_elems * (n - 1)
    return {"bytes": nodes * n * size * (src_elems + dst_elems), "flops": nodes * adds}


def tolerance(case):
    """Sums are binary32 in rank order with one rounding at the end, copies are copies: every bit is determined."""
    return "exact"
