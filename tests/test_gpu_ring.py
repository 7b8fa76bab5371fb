"""Ring schedules with everything left to the library (reductions folded into one chain of additions per
unit, or with their hops in clusters, through shared memory) against the same schedule on the op queues: the same bits, at the edges of tiles and launch shapes."""
import pytest
import torch

from gpu_harness import DT, stream_handle
from paper_2609_36954_b200 import binding as B
from test_gpu_flat import SIZE, same_bits

pytestmark = pytest.mark.gpu


def build(coll, n):
    return lambda c, o: B.pl_schedule_build(c, coll, B.PL_ALGO_RING, n, 64 * 1024, o)


# units (16 bytes) of a partition: a single one, around a warp and the tiles of 64, 128, 256 and 1024
# units, and one large enough for the largest tile with a ragged end
@pytest.mark.parametrize("R,dtype", [(2, "f32"), (2, "i32"), (3, "bf16"), (5, "f32"), (8, "bf16"), (8, "i32"), (16, "bf16"), (16, "f32")])
@pytest.mark.parametrize("units", [1, 31, 33, 257, 4099, 9001, 65539, "large"])
def test_reducing_rings(R, dtype, units):
    units = units if units != "large" else 2 ** 20 // R + 1025
    n = 16 * units // SIZE[dtype] * R
    for coll in (B.PL_REDUCE_SCATTER, B.PL_ALLREDUCE):
        info = same_bits(R, dtype, build(coll, n), "tiles", **({"out_scale": 0.375} if dtype != "i32" else {}))
        assert info.scratch_bytes == 0


@pytest.mark.parametrize("R,dtype", [(2, "i32"), (3, "f32"), (8, "bf16"), (16, "bf16")])
@pytest.mark.parametrize("units", [1, 33, 4099, 65539])
def test_rings_that_keep_their_hops(R, dtype, units):
    """A CTA per rank: the same bits as on the queues, which is what the folded form is compared with above."""
    n = 16 * units // SIZE[dtype] * R
    for coll in (B.PL_REDUCE_SCATTER, B.PL_ALLREDUCE):
        info = same_bits(R, dtype, build(coll, n), "tiles", flags=B.PL_OPT_RING_HOPS)
        assert info.scratch_bytes == 0 and info.grid % R == 0


# up to 1 MiB per rank and 8 MiB in all in clusters, above that on the op queues (two ranks gather without flags: tiles)
@pytest.mark.parametrize("R,dtype", [(2, "f32"), (3, "bf16"), (8, "u8"), (16, "bf16")])
@pytest.mark.parametrize("units", [1, 33, 4099, 32768, 65536, 65537])
def test_gathering_rings(R, dtype, units):
    same_bits(R, dtype, build(B.PL_ALLGATHER, 16 * units // SIZE[dtype]), "tiles" if R == 2 or (units <= 65536 and units * R <= 8 * 65536) else "queues")


def in_clusters(info):
    """Hops through shared memory: a CTA per rank with the tile's slots and nothing else (tiles have none, or a barrier beside them)."""
    return info.smem_bytes > 0 and info.smem_bytes % info.stage_bytes == 0


FORMS = pytest.mark.parametrize("flags", [0, B.PL_OPT_RING_HOPS], ids=["folded", "clusters"])


@FORMS
def test_broken_wait_times_out(flags):
    """The fault hook moves the schedule to the op queues, whose waits it edits."""
    R, n = 4, 4096
    comm = B.pl_comm_create(R, DT["f32"])
    s = build(B.PL_ALLREDUCE, n)(comm, B.make_opts(timeout_ns=20_000_000, flags=flags))
    try:
        assert in_clusters(B.pl_schedule_info(s)) == bool(flags)
        t = [torch.ones(n, device="cuda") for _ in range(2 * R)]
        size = [4 * n] * R
        bufs = B.make_bufs([x.data_ptr() for x in t[:R]], [x.data_ptr() for x in t[R:]], size, size)
        B.pl_execute(s, bufs, stream_handle())
        torch.cuda.synchronize()
        assert all(bool((x == R).all()) for x in t[R:])
        B.pl_schedule_debug_break_wait(s, next(o.topo for o in B.pl_schedule_dump(s) if o.n_wait > 0))
        assert B.pl_schedule_info(s).scratch_bytes > 0
        B.pl_execute(s, bufs, stream_handle())
        torch.cuda.synchronize()
        assert B.pl_comm_status(comm).code == B.PL_ERR_TIMEOUT
    finally:
        B.pl_schedule_destroy(s)
        B.pl_comm_destroy(comm)


@FORMS
def test_a_ring_without_queues_uploads_no_op_list(flags):
    R, n = 16, 32 * 1024 * 1024  # 64 MiB of bf16 per rank in chunks of 64 KiB: 30,720 ops
    comm = B.pl_comm_create(R, DT["bf16"])
    opts = B.make_opts(flags=flags)
    scheds = [build(B.PL_ALLREDUCE, n)(comm, opts)]
    try:
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        scheds += [build(B.PL_ALLREDUCE, n)(comm, opts) for _ in range(6)]
        assert all(in_clusters(B.pl_schedule_info(s)) == bool(flags) for s in scheds)
        assert len(B.pl_schedule_dump(scheds[0])) >= 30720 and B.pl_schedule_info(scheds[0]).scratch_bytes == 0
        assert free - torch.cuda.mem_get_info()[0] < 4 << 20  # an op list takes 3 MiB
    finally:
        for s in scheds:
            B.pl_schedule_destroy(s)
        B.pl_comm_destroy(comm)
