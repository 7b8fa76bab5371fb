"""The rules that pick an executor, on the CPU: the host-only part of the library compiled with g++."""
import ctypes as C
import os
import subprocess
import time

import numpy as np
import pytest

from paper_2609_36954_b200 import binding as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MIB = 1 << 20


@pytest.fixture(scope="session")
def rules(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("rules") / "rules.so")
    csrc = os.path.join(ROOT, "paper_2609_36954_b200", "csrc")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", csrc, "-o", out,
                    os.path.join(csrc, "pl_orchestrator.cpp"), os.path.join(ROOT, "tests", "native", "dispatch_rules.cpp")], check=True)
    L = C.CDLL(out)
    u64, i, u32, p = C.c_uint64, C.c_int, C.c_uint32, C.c_void_p
    L.t_flat_plan.argtypes = [i, i, i, i, u64, u64, p, i, u32, p, i, p, p]
    L.t_queues_faster.argtypes = [i, i, u32, i, i, i, i, u64]
    L.t_ring_folds.argtypes = [i, i, u64]
    L.t_flat_release.argtypes = [i, i, i, i, i, u64]
    L.t_combine_by_parts.argtypes = [u64, u32, i, u64]
    L.t_small_dispatch_rows.argtypes = [i, i, i, i, i, u64]
    L.t_layers.argtypes = [i, u64, i]
    L.t_ring_shape.argtypes = [i, i, i, i, u64, u64, p]
    L.t_flat_run.argtypes = [p, i]
    L.t_ring_plan.argtypes = [i, i, u64, p]
    L.t_validate_changed.argtypes = [i, i, i, i, u64, u64, i, i, i, C.c_char_p, i]
    return L


# MiB of a message, R: a one-shot all-reduce whose inputs do not fit L2 is left to the queues, which read them
# once; one that fits is not.
@pytest.mark.parametrize("R,mib,dtype,hook,queues", [
    (8, 256, "bf16", 0, 1), (8, 16, "bf16", 0, 1), (8, 12, "f32", 0, 1), (8, 8, "bf16", 0, 0), (8, 1, "bf16", 0, 0), (4, 64, "i32", 0, 1),
    (2, 16, "bf16", 0, 0), (16, 5, "bf16", 0, 1), (16, 5, "i32", 0, 0), (16, 6, "i32", 0, 1), (8, 16, "bf16", B.PL_HOOK_RESIDUAL, 1),
    (8, 12, "bf16", B.PL_HOOK_RESIDUAL, 0), (12, 0.75, "bf16", 0, 1), (13, 0.75, "bf16", 0, 0), (16, 0.5, "f32", 0, 1), (16, 1, "bf16", 0, 0),
    (8, 16, "f32", 0, 0), (16, 64, "f32", 0, 0), (12, 6, "f32", 0, 1), (12, 12, "f32", 0, 0), (3, 32, "bf16", 0, 0), (6, 12, "bf16", 0, 0), (6, 16, "bf16", 0, 1),
    (2, 64, "bf16", B.PL_HOOK_RESIDUAL, 0), (14, 16, "bf16", B.PL_HOOK_RESIDUAL, 0), (16, 16, "bf16", B.PL_HOOK_F32_OUT, 0), (8, 16, "bf16", B.PL_HOOK_F32_OUT, 1),
    (16, 16, "bf16", B.PL_HOOK_F32_OUT | B.PL_HOOK_RESIDUAL, 1), (8, 16, "f32", B.PL_HOOK_RESIDUAL, 0), (10, 12, "f32", B.PL_HOOK_RESIDUAL, 1)])
def test_one_shot_all_reduce_stays_on_the_queues_where_they_are_faster(rules, R, mib, dtype, hook, queues):
    dt = {"bf16": B.PL_BF16, "f32": B.PL_F32, "i32": B.PL_I32}[dtype]
    tma = 2 * R * mib * MIB >= 256 * MIB
    assert rules.t_queues_faster(R, dt, hook, B.PL_ALGO_ONESHOT, 1, 0, tma, int(mib * MIB)) == queues
    # the same sizes without a second reading of the inputs
    assert rules.t_queues_faster(R, dt, 0, B.PL_ALGO_DIRECT_FUSED, 1, 1, tma, int(mib * MIB)) == 0


# KiB gathered, R: between 10 and 36 MiB written in all, more than 8 ranks gather on the queues
@pytest.mark.parametrize("R,kib,queues", [(16, 1024, 1), (16, 2048, 1), (16, 512, 0), (16, 8192, 0), (14, 1024, 1), (12, 1024, 1), (8, 2048, 0), (4, 4096, 0)])
def test_all_gather_of_many_ranks_stays_on_the_queues_where_they_are_faster(rules, R, kib, queues):
    for tma in (0, 1):
        assert rules.t_queues_faster(R, B.PL_BF16, 0, B.PL_ALGO_DIRECT, 0, 1, tma, kib << 10) == (queues and not tma)
        assert rules.t_queues_faster(R, B.PL_BF16, 0, B.PL_ALGO_DIRECT, 0, 0, tma, kib << 10) == 0  # all-to-all


# ranks, whether it adds and whether to every rank, CTAs: which grids of the register form release the launch behind them at their start
@pytest.mark.parametrize("R,reduce,every,blocks,release", [
    (8, 1, 1, 1, 0), (8, 1, 1, 512, 0), (8, 1, 1, 1023, 0), (8, 1, 1, 1024, 1), (16, 1, 1, 1 << 20, 1),
    (8, 1, 0, 8, 0), (8, 1, 0, 64, 0), (8, 1, 0, 511, 0), (8, 1, 0, 512, 1),
    (8, 0, 1, 8, 0), (8, 0, 1, 1184, 0), (8, 0, 1, 1280, 1), (4, 0, 1, 1280, 0), (4, 0, 1, 1536, 1), (2, 0, 1, 2048, 0), (2, 0, 1, 3072, 1),
    (8, 0, 0, 1, 1), (8, 0, 0, 300, 1), (8, 0, 0, 4096, 1)])
def test_grids_that_release_the_launch_behind_them(rules, R, reduce, every, blocks, release):
    assert rules.t_flat_release(R, reduce, every, 0, 1, blocks) == release
    assert rules.t_flat_release(R, reduce, every, 0, 0, blocks) == (release or blocks <= 32)  # spans read from memory
    assert rules.t_flat_release(R, reduce, every, 1, 1, blocks)  # bulk copies


# tokens of all ranks, KiB of a row, slots: a combine that reads about 200 MB or more takes whole rows in turn
@pytest.mark.parametrize("tokens,kib,topk,parts", [
    (1024, 32, 8, 0), (4096, 32, 8, 0), (4096, 24, 4, 0), (4096, 14, 8, 0), (1024, 24, 8, 0), (768, 32, 8, 1), (512, 14, 8, 1), (1024, 14, 8, 1),
    (8, 32, 8, 1), (1024, 32, 2, 1), (32768, 4, 8, 1), (32768, 14, 8, 0)])
def test_combine_of_wide_rows_takes_turns(rules, tokens, kib, topk, parts):
    assert rules.t_combine_by_parts(tokens, kib * 64, topk, 592) == parts


# ranks, tokens per rank, slots, KiB of a row -> one launch, plain and deduplicated
@pytest.mark.parametrize("R,T,K,kib,one,one_dedup", [
    (8, 16, 8, 32, 1, 1), (8, 4, 8, 32, 1, 1), (8, 64, 8, 32, 1, 1),
    (8, 64, 8, 14, 1, 1), (8, 16, 8, 14, 1, 1), (8, 128, 8, 14, 1, 1), (8, 129, 8, 14, 0, 0), (8, 256, 2, 4, 1, 1), (8, 384, 2, 4, 1, 0), (2, 1024, 1, 1, 1, 1),
    (8, 8, 8, 80, 0, 0)])
def test_one_launch_dispatch_where_it_is_faster(rules, R, T, K, kib, one, one_dedup):
    rows = rules.t_small_dispatch_rows(0, R, T, K, 256, kib << 10), rules.t_small_dispatch_rows(1, R, T, K, 256, kib << 10)
    assert (rows[0] > 0, rows[1] > 0) == (one, one_dedup)
    assert all(r * K <= 64 and r * (kib << 10) <= 64 << 10 for r in rows)
    assert rules.t_small_dispatch_rows(0, R, T, K, 2048, kib << 10) == 0


# layers whose inputs do not fit L2: nothing is asked ahead, and with many ranks the register executor runs them
@pytest.mark.parametrize("R,mib,hook,executor,ahead", [
    (8, 1, 0, 1, 1), (16, 3, 0, 1, 1), (8, 8, 0, 1, 0), (16, 6, 0, 1, 0), (16, 8, 0, 0, 0), (16, 8, 1, 1, 0), (12, 12, 0, 0, 0), (12, 8, 0, 1, 0), (8, 24, 0, 1, 0)])
def test_layers_that_stream(rules, R, mib, hook, executor, ahead):
    assert rules.t_layers(R, mib * MIB, hook) == executor + 2 * ahead


def ring(rules, R, dtype, coll, nbytes, chunk=MIB):
    reduce, gather = coll != "ag", coll != "rs"
    shape = (C.c_int * 4)()
    part = nbytes // 16 if coll == "ag" else nbytes // R // 16
    smem = rules.t_ring_shape(R, {"bf16": B.PL_BF16, "f32": B.PL_F32, "i32": B.PL_I32, "u8": B.PL_U8}[dtype], reduce, gather, part, chunk, shape)
    return part, smem, list(shape)


# ranks, type, MiB, KiB of a chunk: where the queues run a ring
@pytest.mark.parametrize("R,dtype,coll,mib,kib,clusters", [
    (16, "i32", "ar", 64, 256, 0), (16, "i32", "ar", 64, 1024, 0), (16, "i32", "ar", 64, 64, 1), (16, "i32", "rs", 64, 256, 1), (16, "i32", "ar", 32, 256, 1),
    (9, "i32", "ar", 64, 1024, 0), (8, "i32", "ar", 64, 1024, 1), (16, "f32", "ar", 32, 256, 0), (12, "f32", "ar", 64, 1024, 0), (9, "f32", "ar", 64, 1024, 1), (12, "i32", "ar", 128, 256, 0), (16, "f32", "ar", 16, 64, 1),
    (16, "f32", "ar", 16, 256, 1), (16, "bf16", "ar", 64, 1024, 1), (8, "f32", "ar", 256, 1024, 1), (2, "u8", "ag", 1, 64, 1), (2, "u8", "ag", 2, 64, 0)])
def test_rings_that_stay_on_the_queues(rules, R, dtype, coll, mib, kib, clusters):
    assert (ring(rules, R, dtype, coll, mib * MIB, kib << 10)[1] > 0) == clusters


# ranks, units of a partition: the one hop of two ranks stays in clusters while they are one small CTA per SM
@pytest.mark.parametrize("R,gather,units,folds", [(2, 0, 511, 1), (2, 0, 512, 0), (2, 0, 8192, 0), (2, 0, 9472, 0), (2, 0, 9473, 1), (2, 1, 2048, 1), (3, 0, 2048, 1), (8, 0, 2048, 1)])
def test_the_hop_of_two_ranks_is_kept_where_it_is_faster(rules, R, gather, units, folds):
    assert rules.t_ring_folds(R, gather, units) == folds


@pytest.mark.parametrize("R", [2, 3, 5, 8, 12, 16])
@pytest.mark.parametrize("dtype", ["bf16", "f32", "i32"])
@pytest.mark.parametrize("units", [1, 31, 33, 257, 4099, 65539, 300007])
def test_ring_tiles_cover_the_partition(rules, R, dtype, units):
    for coll in ("rs", "ar"):
        part, smem, (threads, per_thread, tile, grid) = ring(rules, R, dtype, coll, 16 * units * R, 1 << 30)
        assert smem == tile * 16 * 2 * (1 if dtype == "i32" else 2) and smem <= 4 * 256 * 64
        assert threads % 32 == 0 and 32 <= threads <= 256 and tile == threads * per_thread
        assert grid % R == 0 and (grid // R - 1) * tile < part <= grid // R * tile


# schedules whose ops read no output, with one destination or all of them, and one that reads its outputs
@pytest.mark.parametrize("coll,algo,layers", [
    (B.PL_REDUCE_SCATTER, B.PL_ALGO_DIRECT, 0), (B.PL_ALLREDUCE, B.PL_ALGO_DIRECT_FUSED, 0), (B.PL_ALLGATHER, B.PL_ALGO_DIRECT, 0),
    (B.PL_ALLREDUCE, B.PL_ALGO_ONESHOT, 0), (B.PL_ALLREDUCE, B.PL_ALGO_DIRECT_FUSED, 5), (B.PL_ALLREDUCE, B.PL_ALGO_DIRECT, 0)])
def test_validator_sees_outputs_written_twice_or_not_at_all(rules, coll, algo, layers):
    R, n, msg = 4, 4 * 4096, C.create_string_buffer(256)
    for which in (0, 3):
        def check(change):
            return rules.t_validate_changed(R, B.PL_F32, coll, algo, n, 8192, layers, which, change, msg, 256), msg.value.decode()
        assert check(0) == (B.PL_OK, "")
        st, text = check(1)
        assert st == B.PL_ERR_INVALID_SCHEDULE
        assert "overlapping bytes" in text or "flag_need" in text or "topological" in text or "signal" in text, text
        for change in (2, 3):
            st, text = check(change)
            assert st == B.PL_ERR_INVALID_SCHEDULE and ("is covered up to byte" in text or "aligned" in text), text


def test_validating_a_layered_schedule_costs_little():
    """80 layers of 128 KiB on 8 ranks: validation takes about as long as the rest of the build (it took seven times as long)."""
    comm = B.pl_comm_create_planner(8, B.PL_BF16)
    try:
        def build(flags):
            best = []
            for _ in range(5):
                t = time.perf_counter()
                s = B.pl_schedule_build_layers(comm, B.PL_ALGO_AUTO, 65536, 80, B.make_opts(flags=flags))
                best.append(time.perf_counter() - t)
                B.pl_schedule_destroy(s)
            return min(best)
        assert build(0) < 4 * build(B.PL_OPT_SKIP_VALIDATE)
    finally:
        B.pl_comm_destroy(comm)


@pytest.mark.parametrize("R", [2, 3, 4, 8, 16])
def test_gathering_rings_have_one_unit_per_thread(rules, R):
    for units in (1, 127, 4095, 32768, 65536):
        _, smem, (threads, per_thread, tile, _) = ring(rules, R, "u8", "ag", 16 * units)
        assert smem == 0 or (per_thread == 1 and tile == threads)


def landing(R, ops_or_spans, out_units):
    """Where every 16-byte unit of every output comes from: (source rank or 255 for the sum of all, source unit); every unit once."""
    out = [np.full((n, 2), -1, np.int64) for n in out_units]
    for src_off, dst_off, units, src, dst in ops_or_spans:
        for r in (range(R) if dst == 255 else (dst,)):
            at = out[r][dst_off:dst_off + units]
            assert at.shape[0] == units and (at == -1).all()
            at[:, 0] = src
            at[:, 1] = np.arange(src_off, src_off + units)
    assert all((o >= 0).all() for o in out)
    return out


# collectives without flags, over types, odd sizes, empty parts and a processing phase: the spans say of every unit of
# every output what the op list says
@pytest.mark.parametrize("R", [2, 3, 5, 8, 16])
@pytest.mark.parametrize("dtype", ["bf16", "f32", "i32", "u8"])
@pytest.mark.parametrize("units", [1, 7, 129, 1025])
def test_spans_say_what_the_ops_say(rules, R, dtype, units):
    dt, es = {"bf16": (B.PL_BF16, 2), "f32": (B.PL_F32, 4), "i32": (B.PL_I32, 4), "u8": (B.PL_U8, 1)}[dtype]
    vec = 16 // es
    part = units * vec
    v1 = [vec * ((3 * p + units) % 11) for p in range(R)]
    v2 = [[vec * ((5 * p + 7 * r + units) % 13) for r in range(R)] for p in range(R)]
    requests = [(B.PL_ALLGATHER, B.PL_ALGO_DIRECT, part, None, 0), (B.PL_ALLTOALL, B.PL_ALGO_DIRECT, part * R, None, 0),
                (B.PL_ALLTOALLV, B.PL_ALGO_DIRECT, 0, v2, 0), (B.PL_ALLGATHERV, B.PL_ALGO_DIRECT, 0, v1, 0),
                (B.PL_SCATTER, B.PL_ALGO_DIRECT, part, None, 0), (B.PL_GATHER, B.PL_ALGO_DIRECT, part, None, 0)]
    if dtype != "u8":
        requests += [(B.PL_ALLREDUCE, B.PL_ALGO_DIRECT_FUSED, part * R, None, 0), (B.PL_ALLREDUCE, B.PL_ALGO_ONESHOT, part, None, 0),
                     (B.PL_REDUCE_SCATTER, B.PL_ALGO_DIRECT, part * R, None, 0), (B.PL_REDUCE_SCATTERV, B.PL_ALGO_DIRECT, 0, v1, 0)]
    if dtype == "bf16":
        requests += [(B.PL_ALLREDUCE, B.PL_ALGO_DIRECT_FUSED, part * R, None, B.PL_HOOK_F32_OUT | B.PL_HOOK_RESIDUAL),
                     (B.PL_REDUCE_SCATTER, B.PL_ALGO_DIRECT, part * R, None, B.PL_HOOK_F32_OUT)]
    for coll, algo, count, counts, hook in requests:
        comm = B.pl_comm_create_planner(R, dt)
        opts = B.make_opts(hook=hook) if hook else None
        try:
            if counts is not None:
                if sum(np.ravel(counts)) == 0:
                    continue
                s = B.pl_schedule_build_v(comm, coll, algo, counts, 256, opts)
            elif coll in (B.PL_SCATTER, B.PL_GATHER):
                s = B.pl_schedule_build_rooted(comm, coll, R - 1, count, 256, opts)
            else:
                s = B.pl_schedule_build(comm, coll, algo, count, 256, opts)
            info = B.pl_schedule_info(s)
            assert info.n_flags == 0
            out_b = 32 if hook & B.PL_HOOK_F32_OUT else 16  # bytes of an output unit
            out_units = [int(info.out_bytes[r]) // out_b for r in range(R)]
            ops = []
            for o in B.pl_schedule_dump(s):
                copy = o.kind == B.PL_OP_COPY
                if not copy:
                    assert o.n_src == R and all(o.src[k].rank == k and o.src[k].offset == o.src[0].offset for k in range(R))
                nbytes = o.count * (1 if copy else es)
                if nbytes:
                    ops.append((o.src[0].offset // 16, o.dst.offset // out_b, nbytes // 16, o.src[0].rank if copy else 255, 255 if o.dst_bcast & 1 else o.dst.rank))
            flat = np.ravel(counts).astype(np.uint64) if counts is not None else None
            buf, red, every = np.zeros((4096, 5), np.uint64), C.c_int(), C.c_int()
            n = rules.t_flat_plan(R, dt, coll, algo, count, 256, flat.ctypes.data if flat is not None else None, R - 1, hook, buf.ctypes.data, 4096,
                                  C.addressof(red), C.addressof(every))
            assert 0 < n <= 4096 and n <= len(ops)
            spans = [tuple(int(x) for x in row) for row in buf[:n]]
            assert {s_[4] == 255 for s_ in spans} == {bool(every.value)} and {s_[3] == 255 for s_ in spans} == {bool(red.value)}
            for a, b in zip(landing(R, ops, out_units), landing(R, spans, out_units)):
                assert np.array_equal(a, b)
            # a run says the same: what is of equal parts in one row, and nothing with two steps
            run = rules.t_flat_run(buf.ctypes.data, n)
            assert run or coll not in (B.PL_REDUCE_SCATTER, B.PL_ALLGATHER, B.PL_ALLREDUCE, B.PL_SCATTER, B.PL_GATHER)
            assert not run or [tuple(int(x) for x in row) for row in buf[:n]] == spans
            B.pl_schedule_destroy(s)
        finally:
            B.pl_comm_destroy(comm)


def test_ops_with_flags_or_scratch_are_not_laid_out(rules):
    buf, red, every = np.zeros((64, 5), np.uint64), C.c_int(), C.c_int()
    for coll, algo in ((B.PL_ALLREDUCE, B.PL_ALGO_DIRECT), (B.PL_ALLREDUCE, B.PL_ALGO_TREE), (B.PL_REDUCE_SCATTER, B.PL_ALGO_RING), (B.PL_ALLREDUCE, B.PL_ALGO_RING)):
        assert rules.t_flat_plan(4, B.PL_F32, coll, algo, 4096, 1024, None, 0, 0, buf.ctypes.data, 64, C.addressof(red), C.addressof(every)) == -1


# a unit's hops in the op list, followed from rank to rank, name the ranks in the order in which a folded ring adds them
@pytest.mark.parametrize("R", [2, 3, 5, 8, 16])
@pytest.mark.parametrize("dtype", ["bf16", "f32", "i32"])
@pytest.mark.parametrize("units,chunk", [(1, 1 << 20), (7, 32), (65, 256)])
def test_folded_rings_add_in_the_order_of_the_hops(rules, R, dtype, units, chunk):
    dt, es = {"bf16": (B.PL_BF16, 2), "f32": (B.PL_F32, 4), "i32": (B.PL_I32, 4)}[dtype]
    for coll in (B.PL_REDUCE_SCATTER, B.PL_ALLREDUCE):
        comm = B.pl_comm_create_planner(R, dt)
        s = B.pl_schedule_build(comm, coll, B.PL_ALGO_RING, units * 16 // es * R, chunk, None)
        try:
            terms, at = {}, {}  # (rank, buffer, byte offset of an op's destination) -> ranks added so far, first input unit
            for o in B.pl_schedule_dump(s):
                src = [(o.src[k].rank, o.src[k].buf, int(o.src[k].offset)) for k in range(o.n_src)]
                dst = (o.dst.rank, o.dst.buf, int(o.dst.offset))
                terms[dst] = [r for x in src for r in ([x[0]] if x[1] == B.PL_BUF_IN else terms[x])]
                at[dst] = next((x[2] // 16 for x in src if x[1] == B.PL_BUF_IN), None)
                at[dst] = at[src[0]] if at[dst] is None else at[dst]
                n = o.count * (1 if o.kind == B.PL_OP_COPY else es) // 16
                terms[dst + ("units",)] = n
            buf = np.zeros((16, 5), np.uint64)
            assert rules.t_ring_plan(R, coll == B.PL_ALLREDUCE, units, buf.ctypes.data) == R
            covered = [0] * R
            for key, order in terms.items():
                if len(key) != 3 or key[1] != B.PL_BUF_OUT:
                    continue
                rank, _, off = key
                n = terms[key + ("units",)]
                span = next(x for x in buf[:R].astype(np.int64) if x[1] <= off // 16 < x[1] + x[2] and x[4] in (255, rank))
                assert off // 16 + n <= span[1] + span[2] and at[key] - span[0] == off // 16 - span[1]
                assert order == [(span[3] + k) % R for k in range(R)]
                covered[rank] += n
            assert covered == [units * (R if coll == B.PL_ALLREDUCE else 1)] * R
        finally:
            B.pl_schedule_destroy(s)
            B.pl_comm_destroy(comm)
