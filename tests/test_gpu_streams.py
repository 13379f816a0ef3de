"""Batches of one context on streams of their own: a run waits for nothing on another batch's stream."""
import numpy as np
import pytest

import oracle
from test_gpu_blocks import B, random_program  # noqa: F401 (the fixture)
from paper_1211_6193_gb300.workloads import rng

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["plain", "batched"])
@pytest.mark.parametrize("reverse", [False, True])
def test_a_run_does_not_wait_for_another_stream(B, mode, reverse):
    """While a kernel of a second or so holds the first stream, a run enqueued behind it must not hold
    up a run on the second: that one is done while the first stream is still held.  (Any two streams may
    share one of the few hardware queues by chance: the best of three pairs of streams counts.)"""
    import torch
    progs = [random_program(rng.derive(41, i), bdim) for i, bdim in enumerate([33, 64, 96, 128, 257, 512, 640, 1024] * 2)]
    want = oracle.run(progs)

    def done_meanwhile(s1, s2):
        with B.Context(mode=mode) as ctx, ctx.load_programs(progs, s1) as a, ctx.load_programs(progs, s2) as b:
            for batch, s in ((a, s1), (b, s2)):          # (kernels are loaded at their first launch)
                batch.run_and_check(s)
                batch.fetch_reports()
            held = torch.cuda.Event()
            with torch.cuda.stream(s1):
                torch.cuda._sleep(2_000_000_000)
            held.record(s1)
            a.run_and_check(s1)
            b.run_and_check(s2)
            s2.synchronize()
            meanwhile = not held.query()
            for batch in (b, a):
                assert [tuple(int(x) for x in r) for r in batch.fetch_reports()] == want.report_tuples()
                for i, arena in enumerate(batch.fetch_all_memory()):
                    assert np.array_equal(arena, want.arenas[i]), i
        return meanwhile

    for _ in range(3):
        pair = torch.cuda.Stream(), torch.cuda.Stream()
        if done_meanwhile(*(reversed(pair) if reverse else pair)):
            return
    assert False, "every run on the second stream waited for the first"


@pytest.mark.parametrize("mode, options", [("plain", {}), ("plain", {"check_global": True}), ("batched", {}),
                                           ("batched", {"check_global": True}), ("batched", {"use_graph": True})])
def test_a_batch_runs_on_other_streams_than_it_was_loaded_on(B, mode, options):
    """Streams of several priorities in turn, with runs pending on them; one of them captured into a graph
    of the caller's; batches that come and go, so that idle side streams serve the next caller's stream."""
    import torch
    progs = [random_program(rng.derive(43, i), bdim) for i, bdim in enumerate([33, 96, 257, 640])]
    want = oracle.run(progs, **({"check_global": True} if "check_global" in options else {}))

    def same(batch):
        assert [tuple(int(x) for x in r) for r in batch.fetch_reports()] == want.report_tuples()
        for i, arena in enumerate(batch.fetch_all_memory()):
            assert np.array_equal(arena, want.arenas[i]), i

    with B.Context(mode=mode, **options) as ctx:
        for _ in range(3):
            streams = [torch.cuda.Stream(priority=p) for p in (0, -1, 0)] + [torch.cuda.default_stream()]
            with ctx.load_programs(progs, streams[0]) as a, ctx.load_programs(progs, streams[1]) as b:
                for s in streams:
                    for batch in (a, b):
                        batch.run_and_check(s)
                        batch.run_and_check(s)
                        same(batch)
                if "use_graph" in options:
                    continue
                g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
                with torch.cuda.graph(g, stream=s):
                    a.run_and_check(s)
                for _ in range(2):
                    g.replay()
                    torch.cuda.synchronize()
                    same(a)


@pytest.mark.parametrize("mode", ["plain", "batched"])
def test_runs_beside_a_callers_capture(B, mode):
    """While a caller's stream is captured, with one batch's run or two on it, other batches run on the
    streams that all were loaded on, behind pending work and not; the graph is replayed afterwards."""
    import torch
    progs = [random_program(rng.derive(47, i), bdim) for i, bdim in enumerate([33, 96, 257, 640])]
    want = oracle.run(progs)

    def same(batch):
        assert [tuple(int(x) for x in r) for r in batch.fetch_reports()] == want.report_tuples()
        for i, arena in enumerate(batch.fetch_all_memory()):
            assert np.array_equal(arena, want.arenas[i]), i

    s0, s1, s = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Stream()
    with B.Context(mode=mode) as ctx, ctx.load_programs(progs, s0) as a, ctx.load_programs(progs, s0) as b, \
            ctx.load_programs(progs, s1) as c, ctx.load_programs(progs, s0) as d:
        for batch, q in ((a, s0), (b, s0), (c, s1), (d, s0)):
            batch.run_and_check(q)
            same(batch)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            a.run_and_check(s)
            c.run_and_check(s1)
            c.run_and_check(s1)                      # (behind the first)
            b.run_and_check(s)
            d.run_and_check(s0)
        same(c)
        same(d)
        for _ in range(2):
            g.replay()
            torch.cuda.synchronize()
            same(a)
            same(b)
        a.run_and_check(s0)
        same(a)
