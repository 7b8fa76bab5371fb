"""Schedules without flags with everything left to the library (one CTA per tile, no queues) against
the same schedule on the op queues: the same bits, at the edges of tiles, in both forms."""
import pytest
import torch

from gpu_harness import DT, stream_handle
from paper_2609_36954_b200 import binding as B

pytestmark = pytest.mark.gpu
SIZE = {"bf16": 2, "f32": 4, "i32": 4, "u8": 1}
MIB = 1 << 20


def values(nbytes, dtype, gen):
    if dtype in ("bf16", "f32"):
        return torch.randn(nbytes // SIZE[dtype], generator=gen, device="cuda").to({"bf16": torch.bfloat16, "f32": torch.float32}[dtype])
    return torch.randint(0, 256, (nbytes,), generator=gen, device="cuda", dtype=torch.uint8)


def executor(info):
    """What runs a schedule that is not asked for a datapath: "tiles" (one CTA, or one cluster of a ring, per tile) or "queues"."""
    if info.stages == 1:
        assert info.stage_bytes > 0 and info.slice_bytes == 0
        return "tiles"
    assert info.grid == info.n_queues
    return "queues"


def same_bits(R, dtype, build, want, **both):
    """`build` makes a schedule from (comm, opts); runs it as the library picks (`want` says on what) and on the register
    queues, compares all outputs."""
    comm = B.pl_comm_create(R, DT[dtype])
    flat, queues = build(comm, B.make_opts(**both)), build(comm, B.make_opts(datapath=B.PL_DP_LDST, **both))
    try:
        info = B.pl_schedule_info(flat)
        assert executor(info) == want and executor(B.pl_schedule_info(queues)) == "queues"
        gen = torch.Generator(device="cuda").manual_seed(3)
        sizes = [[int(a[r]) for r in range(R)] for a in (info.in_bytes, info.out_bytes, info.aux_bytes)]
        ins = [values(max(16, n), dtype, gen) for n in sizes[0]]
        aux = [values(max(16, n), dtype, gen) for n in sizes[2]]
        outs = []
        for s in (flat, queues):
            out = [torch.full((max(16, n) + 16,), 0x5A, dtype=torch.uint8, device="cuda") for n in sizes[1]]
            bufs = B.make_bufs([t.data_ptr() for t in ins], [t.data_ptr() for t in out], sizes[0], sizes[1], [t.data_ptr() for t in aux], sizes[2])
            for _ in range(2):
                B.pl_execute(s, bufs, stream_handle())
            torch.cuda.synchronize()
            outs.append(out)
        assert B.pl_comm_status(comm).code == B.PL_OK
        for r in range(R):
            assert torch.equal(outs[0][r], outs[1][r]), r   # the 16 bytes behind the output included
            assert bool((outs[0][r][sizes[1][r]:] == 0x5A).all())
        return info
    finally:
        B.pl_schedule_destroy(flat)
        B.pl_schedule_destroy(queues)
        B.pl_comm_destroy(comm)


# units (16 bytes) of a partition: a single one, around 128, 256 and 512 (tiles of the forms), and
# sizes that stream (bulk-copy form) with a ragged end
@pytest.mark.parametrize("R,dtype", [(2, "f32"), (3, "bf16"), (4, "i32"), (5, "f32"), (8, "bf16"), (16, "bf16"), (16, "f32")])
@pytest.mark.parametrize("units", [1, 127, 129, 257, 1025, "stream"])
def test_fixed_size_collectives(R, dtype, units):
    part = 16 * units if units != "stream" else (288 * MIB // (2 * R * R) // 16 + 37) * 16
    n = part // SIZE[dtype]
    for coll, algo, count in ((B.PL_ALLREDUCE, B.PL_ALGO_DIRECT_FUSED, n * R), (B.PL_ALLREDUCE, B.PL_ALGO_ONESHOT, n),
                              (B.PL_REDUCE_SCATTER, B.PL_ALGO_DIRECT, n * R), (B.PL_ALLGATHER, B.PL_ALGO_DIRECT, n),
                              (B.PL_ALLTOALL, B.PL_ALGO_DIRECT, n * R)):
        # one-shot: 9 MiB of inputs on 16 ranks are the queues'
        want = "queues" if algo == B.PL_ALGO_ONESHOT and units == "stream" and R == 16 else "tiles"
        for flags in (0, B.PL_OPT_INPUTS_LAST_USE):
            info = same_bits(R, dtype, lambda c, o: B.pl_schedule_build(c, coll, algo, count, 64 * 1024, o), want, flags=flags)
        if units == "stream" and algo == B.PL_ALGO_DIRECT_FUSED:
            assert info.datapath == B.PL_DP_TMA


@pytest.mark.parametrize("R,dtype", [(2, "bf16"), (4, "f32"), (8, "bf16"), (8, "f32"), (16, "bf16")])
@pytest.mark.parametrize("units", [1, 257, "stream"])
def test_processing_phase(R, dtype, units):
    part = 16 * units if units != "stream" else (288 * MIB // (2 * R * R) // 16 + 37) * 16
    n = part // SIZE[dtype] * R
    hooks = [B.PL_HOOK_RESIDUAL] + ([B.PL_HOOK_F32_OUT, B.PL_HOOK_RESIDUAL | B.PL_HOOK_F32_OUT] if dtype == "bf16" else [])
    for hook in hooks:
        for coll, algo in ((B.PL_ALLREDUCE, B.PL_ALGO_DIRECT_FUSED), (B.PL_REDUCE_SCATTER, B.PL_ALGO_DIRECT)):
            # fused with fp32 output: the queues' up to 8 MiB of inputs, and where it streams without a residual
            f32_fused = algo == B.PL_ALGO_DIRECT_FUSED and hook & B.PL_HOOK_F32_OUT
            want = "queues" if f32_fused and (units != "stream" or hook == B.PL_HOOK_F32_OUT) else "tiles"
            same_bits(R, dtype, lambda c, o: B.pl_schedule_build(c, coll, algo, n, 64 * 1024, o), want, hook=hook, out_scale=0.375)


# units of a partition: 4 x 4 MiB and a ragged end, 16 ranks on both sides of 8 MiB of inputs
@pytest.mark.parametrize("R,units,want", [(4, 65536 + 37, "tiles"), (8, 8192 + 129, "tiles"), (16, 2049, "tiles"), (16, 2048, "queues")])
@pytest.mark.parametrize("hook", [B.PL_HOOK_F32_OUT, B.PL_HOOK_RESIDUAL | B.PL_HOOK_F32_OUT])
def test_fused_with_f32_output_between_its_lines(R, units, want, hook):
    same_bits(R, "bf16", lambda c, o: B.pl_schedule_build(c, B.PL_ALLREDUCE, B.PL_ALGO_DIRECT_FUSED, 8 * units * R, 64 * 1024, o), want, hook=hook, out_scale=0.375)


# MiB of a message above L2 with one-shot, KiB gathered by many ranks
@pytest.mark.parametrize("R,coll,nbytes,want", [
    (8, "oneshot", 16 * MIB, "queues"), (8, "oneshot", 8 * MIB, "tiles"), (3, "oneshot", 32 * MIB // 48 * 48, "tiles"), (16, "gather", MIB, "queues"), (16, "gather", MIB // 2, "tiles"), (12, "gather", 3 * 330 * 1024, "queues")])
def test_sizes_that_stay_on_the_queues(R, coll, nbytes, want):
    n = nbytes // 2
    if coll == "oneshot":
        same_bits(R, "bf16", lambda c, o: B.pl_schedule_build(c, B.PL_ALLREDUCE, B.PL_ALGO_ONESHOT, n, MIB, o), want)
    else:
        same_bits(R, "bf16", lambda c, o: B.pl_schedule_build(c, B.PL_ALLGATHER, B.PL_ALGO_DIRECT, n // R // 8 * 8, MIB, o), want)


@pytest.mark.parametrize("scale", [1, 3000])
def test_variable_sizes_and_rooted(scale):
    R = 8
    counts = [[0 if (p + r) % 3 == 0 else 8 * (1 + (5 * p + 11 * r) % 67) * scale for r in range(R)] for p in range(R)]
    same_bits(R, "bf16", lambda c, o: B.pl_schedule_build_v(c, B.PL_ALLTOALLV, B.PL_ALGO_DIRECT, counts, 4096, o), "tiles")
    for coll in (B.PL_ALLGATHERV, B.PL_REDUCE_SCATTERV):
        same_bits(R, "bf16", lambda c, o: B.pl_schedule_build_v(c, coll, B.PL_ALGO_DIRECT, counts[2], 4096, o), "tiles")
    for coll in (B.PL_BROADCAST, B.PL_REDUCE, B.PL_SCATTER, B.PL_GATHER):
        same_bits(R, "bf16", lambda c, o: B.pl_schedule_build_rooted(c, coll, 5, 8 * R * 77 * scale, 4096, o), "tiles")
    # 256 spans, those between different ranks a single vector
    one = [[8 if p != r else 8 * 50 * scale for r in range(16)] for p in range(16)]
    same_bits(16, "bf16", lambda c, o: B.pl_schedule_build_v(c, B.PL_ALLTOALLV, B.PL_ALGO_DIRECT, one, 4096, o), "tiles")


def test_results_that_fit_l2_stay_there():
    """What a caller reads next must not be the first to leave L2: an all-gather of 8 x 8 MiB and a reader of its
    results take as long as with PL_OPT_NO_L2_HINTS (stored evict-first they took 12 % longer)."""
    R, n = 8, 4 * MIB
    comm = B.pl_comm_create(R, DT["bf16"])
    scheds = [B.pl_schedule_build(comm, B.PL_ALLGATHER, B.PL_ALGO_DIRECT, n // R, MIB, B.make_opts(flags=f)) for f in (0, B.PL_OPT_NO_L2_HINTS)]
    try:
        info = B.pl_schedule_info(scheds[0])
        assert info.datapath == B.PL_DP_LDST and info.grid != info.n_queues
        sets = []
        for _ in range(3):
            x, y = [torch.randn(n // R, device="cuda").bfloat16() for _ in range(R)], torch.empty(R * n, dtype=torch.bfloat16, device="cuda")
            sets.append((x, y, B.make_bufs([t.data_ptr() for t in x], [y[r * n:].data_ptr() for r in range(R)], [2 * n // R] * R, [2 * n] * R)))
        top = torch.empty(64, dtype=torch.bfloat16, device="cuda")
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        times = ([], [])
        for rep in range(12):  # both in turn
            for k, s in enumerate(scheds):
                t0.record()
                for _ in range(20):
                    for _, y, bufs in sets:
                        B.pl_execute(s, bufs, stream_handle())
                        torch.amax(y.view(64, -1), 1, out=top)
                t1.record()
                torch.cuda.synchronize()
                if rep >= 2:
                    times[k].append(t0.elapsed_time(t1))
        default, plain = (sorted(t)[len(t) // 2] for t in times)
        assert default <= 1.06 * plain, (default, plain)
    finally:
        for s in scheds:
            B.pl_schedule_destroy(s)
        B.pl_comm_destroy(comm)


# sums with a second operand have a kernel for a fixed number of ranks: around the ends of warps and tiles, one unit
@pytest.mark.parametrize("R", [2, 3, 4, 5, 6, 8, 12, 16])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("units", [1, 31, 255, 513])
def test_residual_by_number_of_ranks(R, dtype, units):
    n = 16 * units // SIZE[dtype] * R
    for coll, algo in ((B.PL_ALLREDUCE, B.PL_ALGO_DIRECT_FUSED), (B.PL_REDUCE_SCATTER, B.PL_ALGO_DIRECT)):
        for flags in (0, B.PL_OPT_INPUTS_LAST_USE):
            same_bits(R, dtype, lambda c, o: B.pl_schedule_build(c, coll, algo, n, 64 * 1024, o), "tiles", hook=B.PL_HOOK_RESIDUAL, out_scale=0.375, flags=flags)
