"""The work that a user of this library has it do, as cases that can be timed and compared.

A case names a collective (or a fixed sequence of them), the emulated ranks, the element type and
the sizes.  ``prepare`` makes what a program holds before the call (device buffers, communicator,
schedule or plan), ``run`` is one pass through the public entry points of the binding, and ``work``
is what the pass cannot do without: every input byte read once, every output byte written once.
"""
import math

import torch

from paper_2609_36954_b200 import binding as B

KIB, MIB = 1 << 10, 1 << 20
PL_TYPE = {"bf16": B.PL_BF16, "f32": B.PL_F32, "i32": B.PL_I32, "u8": B.PL_U8}
TORCH_TYPE = {"bf16": torch.bfloat16, "f32": torch.float32, "i32": torch.int32, "u8": torch.uint8}
SIZE = {"bf16": 2, "f32": 4, "i32": 4, "u8": 1}


def listed():
    return [
        # One small all-reduce on its own: a decode-sized message outside a layered launch.
        {"name": "allreduce_4kib", "kind": "allreduce", "algo": "auto", "R": 8, "dtype": "bf16", "bytes": 4 * KIB, "chunk": MIB, "residual": False},
        # fp32 gradients or statistics of no round size on three ranks.
        {"name": "allreduce_ragged_f32", "kind": "allreduce", "algo": "auto", "R": 3, "dtype": "f32", "bytes": 3 * (317 * KIB + 16), "chunk": MIB, "residual": False},
        # Tensor-parallel prefill: 1024 tokens x hidden 8192, the residual added before the store.
        {"name": "allreduce_16mib_residual", "kind": "allreduce", "algo": "auto", "R": 8, "dtype": "bf16", "bytes": 16 * MIB, "chunk": MIB, "residual": True},
        # The largest message of the sweep.
        {"name": "allreduce_256mib", "kind": "allreduce", "algo": "auto", "R": 8, "dtype": "bf16", "bytes": 256 * MIB, "chunk": MIB, "residual": False},
        # Ring all-reduce of 262144 fp32 elements per rank in 64 KiB chunks.
        {"name": "ring_allreduce_1mib_f32", "kind": "allreduce", "algo": "ring", "R": 4, "dtype": "f32", "bytes": MIB, "chunk": 64 * KIB, "residual": False},
        # Reduce-scatter in ring order, 64 MiB per rank.
        {"name": "ring_reduce_scatter_64mib", "kind": "reduce_scatter", "algo": "ring", "R": 8, "dtype": "bf16", "bytes": 64 * MIB, "chunk": MIB},
        # The sharded-optimiser step: gradients reduce-scattered, the partitions gathered.
        {"name": "reduce_scatter_all_gather_64mib", "kind": "rs_ag", "R": 8, "dtype": "bf16", "bytes": 64 * MIB, "chunk": MIB},
        # All-to-all of unequal parts: about 24 MiB sent by each rank, Zipf(0.125) shares.
        {"name": "alltoallv_24mib", "kind": "alltoallv", "R": 8, "dtype": "bf16", "bytes": 24 * MIB + 5 * 1040, "chunk": 256 * KIB},
        # Expert parallelism, prefill: 4096 tokens per rank, top-8 of 256 experts, hidden 7168.
        {"name": "moe_prefill_4096", "kind": "moe", "R": 8, "tokens": 4096, "hidden": 7168, "experts": 256, "topk": 8, "dedup": False},
        # Expert parallelism, decode: 64 tokens per rank.
        {"name": "moe_decode_64", "kind": "moe", "R": 8, "tokens": 64, "hidden": 7168, "experts": 256, "topk": 8, "dedup": False},
        # Tensor-parallel decode: 80 layers in one launch, batch 1 and batch 64 x hidden 8192.
        {"name": "decode_80_layers_16kib", "kind": "layers", "R": 8, "dtype": "bf16", "bytes": 16 * KIB, "layers": 80},
        {"name": "decode_80_layers_1mib", "kind": "layers", "R": 8, "dtype": "bf16", "bytes": MIB, "layers": 80},
    ]


def _log_between(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _message(rng, lo, hi, R):
    """Per-rank bytes between lo and hi: half of them powers of two, the others of any size that
    R partitions of 16-byte vectors allow."""
    unit = 16 * R
    n = _log_between(rng, lo, hi)
    if rng.random() < 0.4:
        n = 2 ** round(math.log2(n))
    return max(unit, int(n) // unit * unit)


def draw(rng):
    kind = rng.choice(["allreduce", "allreduce", "allreduce", "ring", "ring", "rs_ag", "alltoallv", "moe", "moe", "layers", "layers"])
    if kind == "allreduce":
        R = rng.choice([2, 3, 4, 6, 8, 8, 8, 16])
        dtype = rng.choice(["bf16", "bf16", "bf16", "f32", "i32"])
        residual = dtype != "i32" and rng.random() < 0.3
        hi = min(256 * MIB, (768 if residual else 2048) * MIB // R)
        return {"kind": kind, "algo": "auto", "R": R, "dtype": dtype, "bytes": _message(rng, KIB, hi, R), "chunk": MIB, "residual": residual}
    if kind == "ring":
        R = rng.choice([2, 4, 4, 8, 8])
        case = {"kind": rng.choice(["allreduce", "reduce_scatter"]), "algo": "ring", "R": R, "dtype": rng.choice(["bf16", "f32", "i32"]),
                "bytes": _message(rng, 64 * KIB, 64 * MIB, R), "chunk": rng.choice([64 * KIB, 256 * KIB, MIB])}
        if case["kind"] == "allreduce":
            case["residual"] = False
        return case
    if kind == "rs_ag":
        R = rng.choice([2, 4, 8, 8])
        return {"kind": kind, "R": R, "dtype": rng.choice(["bf16", "bf16", "f32"]), "bytes": _message(rng, 256 * KIB, 128 * MIB, R), "chunk": rng.choice([256 * KIB, MIB])}
    if kind == "alltoallv":
        return {"kind": kind, "R": rng.choice([4, 8, 8]), "dtype": rng.choice(["bf16", "f32", "u8"]), "bytes": int(_log_between(rng, 64 * KIB, 128 * MIB)), "chunk": rng.choice([256 * KIB, MIB])}
    if kind == "moe":
        return {"kind": kind, "R": rng.choice([4, 8, 8]), "tokens": max(1, int(_log_between(rng, 1, 4096))), "hidden": rng.choice([512, 2048, 4096, 7168]),
                "experts": rng.choice([32, 64, 256]), "topk": rng.choice([2, 4, 6, 8]), "dedup": rng.random() < 0.3}
    R = rng.choice([4, 8, 8])
    return {"kind": kind, "R": R, "dtype": rng.choice(["bf16", "bf16", "f32"]), "bytes": _message(rng, 4 * KIB, MIB, R), "layers": rng.randint(16, 80)}


class _Comm:
    """A communicator with the schedules and plans built on it, given back with the state."""

    def __init__(self, R, dtype):
        self.comm, self.schedules, self.plans = B.pl_comm_create(R, dtype), [], []

    def schedule(self, handle):
        self.schedules.append(handle)
        return handle

    def plan(self, handle):
        self.plans.append(handle)
        return handle

    def __del__(self):
        for s in self.schedules:
            B.pl_schedule_destroy(s)
        for p in self.plans:
            B.pl_moe_plan_destroy(p)
        B.pl_comm_destroy(self.comm)


def _values(n, dtype, gen):
    """Activations and gradients ~ N(0, 1); whole numbers over a range whose sums stay exact; any byte."""
    if dtype in ("bf16", "f32"):
        return torch.randn(n, generator=gen, device="cuda", dtype=torch.float32).to(TORCH_TYPE[dtype])
    if dtype == "i32":
        return torch.randint(-(1 << 24), 1 << 24, (n,), generator=gen, device="cuda", dtype=torch.int32)
    return torch.randint(0, 256, (n,), generator=gen, device="cuda", dtype=torch.uint8)


def _empty(nbytes, dtype):
    return torch.empty(int(nbytes) // SIZE[dtype], device="cuda", dtype=TORCH_TYPE[dtype])


def _ptrs(tensors):
    return [t.data_ptr() for t in tensors]


def _bufs(info, ins, outs, aux=None):
    R = len(ins)
    if aux is None:
        return B.make_bufs(_ptrs(ins), _ptrs(outs), list(info.in_bytes)[:R], list(info.out_bytes)[:R])
    return B.make_bufs(_ptrs(ins), _ptrs(outs), list(info.in_bytes)[:R], list(info.out_bytes)[:R], _ptrs(aux), list(info.aux_bytes)[:R])


def _alltoallv_counts(case):
    """Elements sent from p to r.  Rank r's share of a message is ~ (r + 1) ** -0.125, rotated from
    source to source so that every rank sends and receives about the same, in 16-byte vectors."""
    R, per = case["R"], 16 // SIZE[case["dtype"]]
    w = [(r + 1.0) ** -0.125 for r in range(R)]
    share = [int(case["bytes"] * v / sum(w)) // 16 * per for v in w]
    return [[share[(r - p - 1) % R] for r in range(R)] for p in range(R)]


def _routing(case, gen):
    """Top-k distinct experts per token with Zipf(1.2) popularity (Gumbel top-k over a shuffled
    popularity order, the same for every seed as it is for a model) and the fp32 softmax of the
    selected logits as gates."""
    R, T, E, K = case["R"], case["tokens"], case["experts"], case["topk"]
    logp = -1.2 * torch.log(torch.arange(1, E + 1, device="cuda", dtype=torch.float32))
    logp = logp[torch.randperm(E, generator=torch.Generator().manual_seed(1)).cuda()]
    noise = torch.rand(R * T, E, generator=gen, device="cuda").clamp_(1e-9, 1 - 1e-7)
    top, idx = torch.topk(logp - torch.log(-torch.log(noise)), K, dim=1)
    gates = torch.softmax(top, dim=1)
    return ([t.contiguous() for t in idx.to(torch.int32).view(R, T, K).unbind(0)],
            [t.contiguous() for t in gates.view(R, T, K).unbind(0)])


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    stream = torch.cuda.current_stream().cuda_stream
    kind, R = case["kind"], case["R"]
    if kind == "moe":
        return _prepare_moe(case, gen, stream)
    dtype = case["dtype"]
    own = _Comm(R, PL_TYPE[dtype])
    n = case["bytes"] // SIZE[dtype]
    state = {"kind": kind, "own": own, "stream": stream}
    if kind == "alltoallv":
        counts = _alltoallv_counts(case)
        s = own.schedule(B.pl_schedule_build_v(own.comm, B.PL_ALLTOALLV, B.PL_ALGO_DIRECT, counts, case["chunk"]))
    elif kind == "layers":
        s = own.schedule(B.pl_schedule_build_layers(own.comm, B.PL_ALGO_AUTO, n, case["layers"]))
    elif kind == "rs_ag":
        # Both launches read their inputs for the last time, and the reduce-scatter may be set up
        # while the all-gather of the step before drains.
        last_use = B.make_opts(flags=B.PL_OPT_INPUTS_LAST_USE)
        s = own.schedule(B.pl_schedule_build(own.comm, B.PL_REDUCE_SCATTER, B.PL_ALGO_DIRECT, n, case["chunk"],
                                             B.make_opts(flags=B.PL_OPT_INPUTS_LAST_USE | B.PL_OPT_OVERLAP_LAUNCH)))
        g = own.schedule(B.pl_schedule_build(own.comm, B.PL_ALLGATHER, B.PL_ALGO_DIRECT, n // R, case["chunk"], last_use))
    else:
        coll = B.PL_ALLREDUCE if kind == "allreduce" else B.PL_REDUCE_SCATTER
        algo = B.PL_ALGO_RING if case["algo"] == "ring" else B.PL_ALGO_AUTO
        opts = B.make_opts(hook=B.PL_HOOK_RESIDUAL) if case.get("residual") else None
        s = own.schedule(B.pl_schedule_build(own.comm, coll, algo, n, case["chunk"], opts))
    info = B.pl_schedule_info(s)
    ins = [_values(int(info.in_bytes[r]) // SIZE[dtype], dtype, gen) for r in range(R)]
    outs = [_empty(info.out_bytes[r], dtype) for r in range(R)]
    aux = [_values(int(info.aux_bytes[r]) // SIZE[dtype], dtype, gen) for r in range(R)] if case.get("residual") else None
    state.update(schedule=s, ins=ins, outs=outs, aux=aux, bufs=_bufs(info, ins, outs, aux))
    if kind == "rs_ag":
        gathered = B.pl_schedule_info(g)
        full = [_empty(gathered.out_bytes[r], dtype) for r in range(R)]
        state.update(gather=g, full=full, gather_bufs=_bufs(gathered, outs, full))
    return state


def _prepare_moe(case, gen, stream):
    R, T, H, E, K = case["R"], case["tokens"], case["hidden"], case["experts"], case["topk"]
    idx, gates = _routing(case, gen)
    # receive buffers for up to three times the mean load of a rank (the routing is skewed)
    rows = min(R * T * K, 3 * T * K + 64)
    own = _Comm(R, B.PL_BF16)
    plan = own.plan(B.pl_moe_plan_create(own.comm, T, H, E, K, rows))
    x = [_values(T * H, "bf16", gen).view(T, H) for _ in range(R)]
    y = [_values(rows * H, "bf16", gen).view(rows, H) for _ in range(R)]  # what the experts made of their rows
    recv = [torch.zeros(rows, H, device="cuda", dtype=torch.bfloat16) for _ in range(R)]
    meta = [torch.zeros(rows, 4, device="cuda", dtype=torch.int32) for _ in range(R)]
    out = [torch.empty(T, H, device="cuda", dtype=torch.bfloat16) for _ in range(R)]
    return {"kind": "moe", "own": own, "stream": stream, "plan": plan, "dedup": case["dedup"], "x": x, "idx": idx, "gates": gates,
            "y": y, "recv": recv, "meta": meta, "out": out, "at": {"x": _ptrs(x), "idx": _ptrs(idx), "gates": _ptrs(gates),
                                                          "y": _ptrs(y), "recv": _ptrs(recv), "meta": _ptrs(meta), "out": _ptrs(out)}}


def run(state):
    stream = state["stream"]
    if state["kind"] == "moe":
        # tokens to their experts, and the experts' results back (the experts are not part of it)
        plan, at = state["plan"], state["at"]
        if state["dedup"]:
            B.pl_moe_dispatch_dedup(plan, at["x"], at["idx"], at["recv"], at["meta"], stream)
            B.pl_moe_combine_dedup(plan, at["y"], at["out"], stream)
        else:
            B.pl_moe_dispatch(plan, at["x"], at["idx"], at["recv"], at["meta"], stream)
            B.pl_moe_combine(plan, at["y"], at["gates"], at["out"], stream)
        return {"recv": state["recv"], "meta": state["meta"], "out": state["out"]}
    B.pl_execute(state["schedule"], state["bufs"], stream)
    if state["kind"] == "rs_ag":
        B.pl_execute(state["gather"], state["gather_bufs"], stream)
        return {"partitions": state["outs"], "gathered": state["full"]}
    return state["outs"]


def work(case):
    R, kind = case["R"], case["kind"]
    if kind == "moe":
        T, K, row = case["tokens"], case["topk"], case["hidden"] * 2
        # rows sent: one per token and expert, or per token and rank that holds one of its experts
        # (about what a uniform choice of the ranks gives)
        rows = R * T * (R * (1 - (1 - 1 / R) ** K) if case["dedup"] else K)
        index = R * T * K * (4 if case["dedup"] else 8)
        return {"bytes": 2 * R * T * row + 2 * rows * row + 16 * rows + index, "flops": 2 * rows * case["hidden"]}
    m = case["bytes"]
    n = m // SIZE[case["dtype"]]
    if kind == "alltoallv":
        return {"bytes": 2 * SIZE[case["dtype"]] * sum(map(sum, _alltoallv_counts(case))), "flops": 0}
    if kind == "layers":
        return {"bytes": case["layers"] * 2 * R * m, "flops": case["layers"] * (R - 1) * n}
    if kind == "rs_ag":
        return {"bytes": 2 * R * m + m, "flops": (R - 1) * n}
    if kind == "reduce_scatter":
        return {"bytes": R * m + m, "flops": (R - 1) * n}
    return {"bytes": (3 if case["residual"] else 2) * R * m, "flops": ((R if case["residual"] else 0) + R - 1) * n}


def tolerance(case):
    if case["kind"] == "alltoallv" or case.get("dtype") == "i32":
        return "exact"
    if case.get("dtype") == "f32":
        # measured: 3e-8 off the sum in 64 bits, 5e-8 off (1.9e-7 .. 2.3e-7 at most) another order of the sum
        return {"rel": 4e-7, "max": 4e-6}
    # measured: 1.7e-3 off the sum in 64 bits, 3.9e-3 at most, both from the one rounding to bf16
    return {"rel": 7e-3, "max": 1.5e-2}
