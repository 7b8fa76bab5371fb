"""Launches that the library sets up while the launch in front drains (the default of every executor here): each
reads what the one in front wrote, in the same buffers turn after turn, so a kernel that looked too early would see the turn
before.  Back to back, in a CUDA graph, behind a fork and join, and several executors at once on streams of their own."""
import numpy as np
import pytest
import torch

from gpu_harness import Session, poison, stream_handle, to_dev
from paper_2609_36954_b200 import binding as B

pytestmark = pytest.mark.gpu
R, LAYERS = 4, 2


def in_clusters(info):
    """A ring that hops through shared memory: the tile's slots of a CTA per rank and nothing else (tiles have none, or a barrier beside them)."""
    return info.smem_bytes > 0 and info.smem_bytes % info.stage_bytes == 0 and info.grid % R == 0


class Chain:
    """x -> fused all-reduce (tiles) -> ring (clusters and, every second turn, folded) -> two layers (`n` decides: one cluster, or flags) -> reduce-scatter
    (tiles) -> all-gather (tiles); with the sum S of the inputs the result is R^3 S on every rank."""

    def __init__(self, n, turns):
        self.ses, self.n = Session(R, "i32"), n
        a = self.ses.build(B.PL_ALLREDUCE, B.PL_ALGO_DIRECT_FUSED, n, 1 << 20)
        b = [self.ses.build(B.PL_ALLREDUCE, B.PL_ALGO_RING, n, 65536, flags=f) for f in (B.PL_OPT_RING_HOPS, 0)]
        c = self.ses.build_layers(B.PL_ALGO_AUTO, n // LAYERS, LAYERS)
        d = self.ses.build(B.PL_REDUCE_SCATTER, B.PL_ALGO_DIRECT, n, 1 << 20)
        e = self.ses.build(B.PL_ALLGATHER, B.PL_ALGO_DIRECT, n // R, 1 << 20)
        for s in (a, *b, d, e):
            assert B.pl_schedule_info(s).stages == 1  # not on the queues
        assert [in_clusters(B.pl_schedule_info(s)) for s in b] == [True, False]
        rng = np.random.default_rng(n)
        x = [rng.integers(-2 ** 31, 2 ** 31, (turns, n)).astype(np.int32) for _ in range(R)]
        with np.errstate(over="ignore"):
            self.want = [(sum(v[t].astype(np.int64) for v in x) * R ** 3).astype(np.int32) for t in range(turns)]
        dx = [[to_dev(v[t]) for v in x] for t in range(turns)]
        y, z, w = ([poison(4 * n) for _ in range(R)] for _ in range(3))
        u = [poison(4 * n // R) for _ in range(R)]
        self.out = [[poison(4 * n) for _ in range(R)] for _ in range(turns)]
        self.keep = (dx, y, z, w, u)

        def bufs(s, i, o):
            info = B.pl_schedule_info(s)
            return s, B.make_bufs([t.data_ptr() for t in i], [t.data_ptr() for t in o], list(info.in_bytes)[:R], list(info.out_bytes)[:R])

        self.calls = [[bufs(a, dx[t], y), bufs(b[t % 2], y, z), bufs(c, z, w), bufs(d, w, u), bufs(e, u, self.out[t])] for t in range(turns)]

    def run(self):
        for turn in self.calls:
            for s, b in turn:
                B.pl_execute(s, b, stream_handle())

    def check(self):
        torch.cuda.synchronize()
        assert B.pl_comm_status(self.ses.comm).code == B.PL_OK
        for t, want in enumerate(self.want):
            for r in range(R):
                assert np.array_equal(self.out[t][r].cpu().numpy().view(np.int32), want), (t, r)
        for o in self.out:
            for t in o:
                t.fill_(0xFF)


# a few KiB (the layers run as one cluster), 1 MiB (with flags)
@pytest.mark.parametrize("n", [64 * R, 2048 * R, 65536 * R])
@pytest.mark.parametrize("how", ["back to back", "graph", "fork and join"])
def test_each_launch_sees_what_the_one_in_front_wrote(n, how):
    c = Chain(n, turns=5)
    try:
        if how == "back to back":
            for _ in range(4):
                c.run()
                c.check()
            return
        g, main, side = torch.cuda.CUDAGraph(), torch.cuda.Stream(), torch.cuda.Stream()
        other = [torch.zeros(1 << 18, device="cuda") for _ in range(2)]
        main.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(g, stream=main):
            if how == "graph":
                c.run()
            else:  # the launch behind a join has two in front of it
                for turn in c.calls:
                    for s, b in turn:
                        side.wait_stream(main)
                        with torch.cuda.stream(side):
                            other[0].add_(1.0)
                        other[1].add_(1.0)
                        main.wait_stream(side)
                        B.pl_execute(s, b, stream_handle())
        for _ in range(3):
            g.replay()
            c.check()
    finally:
        c.ses.close()


def test_executors_whose_launches_wait_for_nobody_run_beside_one_another():
    """Tiles, rings and cluster layers on three streams at once, grids larger than the GPU."""
    n = 1 << 20
    ses = Session(R, "i32")
    try:
        scheds = [ses.build(B.PL_ALLREDUCE, B.PL_ALGO_DIRECT_FUSED, n, 1 << 20),
                  ses.build(B.PL_ALLREDUCE, B.PL_ALGO_RING, n, 65536, flags=B.PL_OPT_RING_HOPS), ses.build_layers(B.PL_ALGO_AUTO, 1024, 8)]
        assert in_clusters(B.pl_schedule_info(scheds[1]))
        assert B.pl_schedule_info(scheds[0]).grid + B.pl_schedule_info(scheds[1]).grid > 1000 and B.pl_schedule_info(scheds[2]).grid <= 16
        jobs = []
        for s in scheds:
            info = B.pl_schedule_info(s)
            x = [torch.randint(-99, 99, (int(info.in_bytes[r]) // 4,), dtype=torch.int32, device="cuda") for r in range(R)]
            y = [poison(info.out_bytes[r]) for r in range(R)]
            jobs.append((s, B.make_bufs([t.data_ptr() for t in x], [t.data_ptr() for t in y], list(info.in_bytes)[:R], list(info.out_bytes)[:R]), x, y, torch.cuda.Stream()))
        torch.cuda.synchronize()
        for _ in range(40):
            for s, b, _, _, st in jobs:
                B.pl_execute(s, b, st.cuda_stream)
        torch.cuda.synchronize()
        assert B.pl_comm_status(ses.comm).code == B.PL_OK
        for _, _, x, y, _ in jobs:
            want = sum(x[1:], x[0].clone())
            assert all(torch.equal(t.view(torch.int32), want) for t in y)
    finally:
        ses.close()
