"""Layered direct-fused all-reduces with the grid left to the library (the layer executor): both
forms of its layer-to-layer join, at the edges of its slices and of the choice between the forms."""
import numpy as np
import pytest
import torch

from gpu_harness import Session, check_float, poison, stream_handle, to_dev
from oracle import oracle
from paper_2609_36954_b200 import binding as B
from paper_2609_36954_b200 import inputs as gen

pytestmark = pytest.mark.gpu
SIZE = {"bf16": 2, "f32": 4, "i32": 4}


def as_f64(raw, dtype):
    return gen.bf16_bits_to_f64(raw.view(np.uint16)) if dtype == "bf16" else raw.view(np.float32).astype(np.float64)


# bytes of a rank's message: one vector per partition, two, a line and a vector, an odd number of
# lines, the last size that runs as one cluster (R * bytes = 256 KiB) and the first that does not,
# more units per slice than threads, the lines of the next layer asked for and (from 64 MiB of inputs) not
@pytest.mark.parametrize("R,dtype,nbytes", [
    (8, "bf16", 128), (8, "bf16", 8 * 32), (8, "i32", 8 * 144), (3, "bf16", 3 * 16 * 37), (8, "bf16", 32768), (8, "bf16", 32768 + 128),
    (2, "f32", 131072), (2, "f32", 131072 + 32), (16, "bf16", 16384), (16, "i32", 16384 + 256), (5, "f32", 5 * 16 * 1001),
    (4, "bf16", 4 << 20), (4, "bf16", (16 << 20) + 64 * 5)])
def test_layers_match_oracle(R, dtype, nbytes):
    n, layers = nbytes // SIZE[dtype], 3
    x = [np.concatenate([gen.rank_inputs(R, n, dtype, seed=l)[r] for l in range(layers)]) for r in range(R)]
    ses = Session(R, dtype)
    try:
        s = ses.build_layers(B.PL_ALGO_DIRECT_FUSED, n, layers)
        for rep in range(2):  # the second execute finds the flags of the first
            outs, _ = ses.execute(s, x, repeats=1 + rep)
            for l in range(layers):
                ref = oracle.allreduce([a[l * n:(l + 1) * n] for a in x], dtype)
                for r in range(R):
                    if dtype == "i32":
                        assert np.array_equal(outs[r].view(np.int32)[l * n:(l + 1) * n], ref[r])
                    else:
                        check_float(as_f64(outs[r], dtype)[l * n:(l + 1) * n], ref[r], dtype)
            x = [np.roll(a, 3) for a in x]
    finally:
        ses.close()


@pytest.mark.parametrize("R,nbytes", [(8, 4096), (8, 65536), (3, 3 * 16 * 37), (16, 65536)])
def test_layers_with_residual_and_f32_output(R, nbytes):
    # fp32 output of equal inputs is exactly R * x + x: no rounding for these small whole numbers
    n, layers = nbytes // 2, 3
    v = np.arange(n * layers) % 97
    x = gen.f32_to_bf16_bits(v.astype(np.float32))
    ses = Session(R, "bf16")
    try:
        s = ses.build_layers(B.PL_ALGO_DIRECT_FUSED, n, layers, hook=B.PL_HOOK_RESIDUAL | B.PL_HOOK_F32_OUT)
        info = B.pl_schedule_info(s)
        d_in, d_aux = [to_dev(x) for _ in range(R)], [to_dev(x) for _ in range(R)]
        d_out = [poison(info.out_bytes[r]) for r in range(R)]
        sizes = [[int(a[r]) for r in range(R)] for a in (info.in_bytes, info.out_bytes, info.aux_bytes)]
        bufs = B.make_bufs([t.data_ptr() for t in d_in], [t.data_ptr() for t in d_out], sizes[0], sizes[1],
                           [t.data_ptr() for t in d_aux], sizes[2])
        B.pl_execute(s, bufs, stream_handle())
        torch.cuda.synchronize()
        assert B.pl_comm_status(ses.comm).code == B.PL_OK
        for r in range(R):
            assert np.array_equal(d_out[r].cpu().numpy().view(np.float32), ((R + 1) * v).astype(np.float32))
    finally:
        ses.close()


@pytest.mark.parametrize("nbytes", [8192, 131072])
def test_layers_trace_and_time_out(nbytes):
    R, n, layers = 8, nbytes // 2, 4
    x = [np.concatenate([gen.normal_bf16(n, 1, l * R + r) for l in range(layers)]) for r in range(R)]
    ses = Session(R, "bf16")
    try:
        s = ses.build_layers(B.PL_ALGO_DIRECT_FUSED, n, layers, flags=B.PL_OPT_TRACE)
        ses.execute(s, x)
        ops = B.pl_schedule_dump(s)
        stamps = B.pl_schedule_trace_read(s, len(ops), stream_handle())
        for l in range(1, layers):  # no op of a layer starts before every op of the layer in front has ended
            ends = max(stamps[o.topo, 1] for o in ops if o.layer == l - 1)
            assert ends and ends <= min(stamps[o.topo, 0] for o in ops if o.layer == l)
        bad = ses.build_layers(B.PL_ALGO_DIRECT_FUSED, n, layers, timeout_ns=20_000_000)
        victim = next(o.topo for o in B.pl_schedule_dump(bad) if o.layer == layers - 1)  # nobody waits behind it
        B.pl_schedule_debug_break_wait(bad, victim)
        with pytest.raises(AssertionError, match="device status 6"):
            ses.execute(bad, x)
        assert B.pl_comm_status(ses.comm).op == victim
        B.pl_comm_reset(ses.comm, stream_handle())
        torch.cuda.synchronize()
        ses.execute(s, x)
    finally:
        ses.close()


# the kernels for a number of ranks and the one for any other, as they ship: every CTA of an execute waits for signals of
# one that never ran, gives up, and says so; after a reset the schedule runs again
@pytest.mark.parametrize("R,dtype", [(8, "bf16"), (9, "f32"), (16, "i32")])
def test_layers_that_time_out_in_the_kernel_that_ships(R, dtype):
    n, layers = 16 * 1024 * R // SIZE[dtype], 4
    ses = Session(R, dtype)
    try:
        s = ses.build_layers(B.PL_ALGO_DIRECT_FUSED, n, layers, timeout_ns=20_000_000)
        assert B.pl_schedule_info(s).grid > 16  # with flags
        x = [(np.arange(n * layers) % 89 + r).astype(np.int32) for r in range(R)]
        x = [gen.f32_to_bf16_bits(a.astype(np.float32)) if dtype == "bf16" else a.astype(np.float32 if dtype == "f32" else np.int32) for a in x]
        want, _ = ses.execute(s, x, repeats=2)
        B.pl_schedule_debug_raise_epoch(s)
        with pytest.raises(AssertionError, match="device status 6"):
            ses.execute(s, x)
        st = B.pl_comm_status(ses.comm)
        grid = B.pl_schedule_info(s).grid
        # third execute, counted as the fourth; layer 1 waits for layer 0, which all CTAs have written
        assert st.expected == 4 * grid and st.observed == 3 * grid and B.pl_schedule_dump(s)[st.op].layer == 1
        B.pl_comm_reset(ses.comm, stream_handle())
        torch.cuda.synchronize()
        again, _ = ses.execute(s, x, repeats=2)
        assert all(np.array_equal(a, b) for a, b in zip(want, again))
        for other in (ses.build_layers(B.PL_ALGO_DIRECT_FUSED, 64 * R, layers), ses.build(B.PL_ALLREDUCE, B.PL_ALGO_DIRECT_FUSED, n, 1 << 20)):
            with pytest.raises(B.PurlinError):  # one cluster; tiles: no epoch of this kind
                B.pl_schedule_debug_raise_epoch(other)
    finally:
        ses.close()


# tiny messages with everything left to the library: the layer executor where the message has a vector for
# every rank, packets where it has not; the same bits as packets asked for
@pytest.mark.parametrize("R,dtype,nbytes,want", [
    (8, "bf16", 128, B.PL_DP_LDST), (8, "bf16", 128 + 16, B.PL_DP_PACKET), (8, "f32", 4096, B.PL_DP_LDST), (3, "f32", 48, B.PL_DP_LDST),
    (3, "bf16", 4096, B.PL_DP_PACKET), (16, "i32", 256, B.PL_DP_LDST), (16, "bf16", 240, B.PL_DP_PACKET), (2, "i32", 4096, B.PL_DP_LDST)])
def test_tiny_layers_left_to_the_library(R, dtype, nbytes, want):
    n, layers = nbytes // SIZE[dtype], 5
    x = [np.concatenate([gen.rank_inputs(R, n, dtype, seed=l)[r] for l in range(layers)]) for r in range(R)]
    ses = Session(R, dtype)
    try:
        auto = ses.build_layers(B.PL_ALGO_AUTO, n, layers)
        assert B.pl_schedule_info(auto).datapath == want
        a, _ = ses.execute(auto, x)
        b, _ = ses.execute(ses.build_layers(B.PL_ALGO_ONESHOT, n, layers, datapath=B.PL_DP_PACKET), x)
        assert all(np.array_equal(p, q) for p, q in zip(a, b))
    finally:
        ses.close()


def test_layers_of_many_ranks_that_stream_run_on_the_register_executor():
    R, n, layers = 16, 4 << 20, 2  # 8 MiB of bf16 per rank: 128 MiB of inputs a layer
    ses = Session(R, "bf16")
    try:
        s = ses.build_layers(B.PL_ALGO_AUTO, n, layers)
        assert len(B.pl_schedule_dump(s)) > layers * B.pl_schedule_info(s).n_queues  # the layer executor has one op per queue and layer
        x = [torch.randint(-8, 8, (layers * n,), device="cuda").bfloat16() for _ in range(R)]
        y = [poison(2 * layers * n) for _ in range(R)]
        size = [2 * layers * n] * R
        B.pl_execute(s, B.make_bufs([t.data_ptr() for t in x], [t.data_ptr() for t in y], size, size), stream_handle())
        torch.cuda.synchronize()
        assert B.pl_comm_status(ses.comm).code == B.PL_OK
        want = sum(t.float() for t in x).bfloat16()  # whole numbers: exact
        assert all(torch.equal(t.view(torch.bfloat16), want) for t in y)
    finally:
        ses.close()


# kernels for a fixed number of ranks, and the one for any other: slices that do not fill a warp, end inside one, and take
# several turns of a thread, as one cluster and with flags, against the register executor (a grid asked for): the same bits
@pytest.mark.parametrize("R", [2, 3, 4, 5, 6, 7, 8, 9, 12, 16])
@pytest.mark.parametrize("dtype", ["bf16", "f32", "i32"])
@pytest.mark.parametrize("units", [1, 33, 149, 2055])
def test_layers_by_number_of_ranks(R, dtype, units):
    layers, es = 3, SIZE[dtype]
    n = 16 * units * R // es
    ses = Session(R, dtype)
    try:
        x = [torch.randn(n * layers, device="cuda", generator=torch.Generator("cuda").manual_seed(r)) for r in range(R)]
        x = [(t * 2 ** 30).to(torch.int32) if dtype == "i32" else t.to(torch.bfloat16 if dtype == "bf16" else torch.float32) for t in x]
        outs, threads = [], []
        for kw in ({}, {"n_ctas": R}):
            s = ses.build_layers(B.PL_ALGO_DIRECT_FUSED, n, layers, **kw)
            outs.append(ses.execute(s, None, repeats=2, d_ins=x)[0])
            threads.append(B.pl_schedule_info(s).threads)
        assert threads[0] < 512 == threads[1]  # as many as a slice needs here, the default of the queues there
        for a, b in zip(*outs):
            assert np.array_equal(a, b)
    finally:
        ses.close()
