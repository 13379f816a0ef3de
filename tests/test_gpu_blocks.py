"""GPU parity at the edges of the interpreter's shapes: block sizes around the limits of the
simulated warps per warp (64, 128) and ragged ones, random kernels whose threads part, join,
collide, leave their arrays and divide by zero, under every optional check; and the report
compaction around the size where it takes one kernel.  Everything is compared with the oracle
bit for bit."""
import numpy as np
import pytest

import oracle
from paper_1211_6193_gb300.workloads import rng
from paper_1211_6193_gb300.workloads.ir import (BID, R, TID, Asm, Launch, Program, r0, r1, r2, r3, r4, r5, r9, r10, r11,
                                                r12)

pytestmark = pytest.mark.gpu

BDIMS = [1, 31, 33, 63, 64, 65, 96, 97, 127, 128, 129, 160, 255, 257, 513, 1000, 1024]
OPTIONS = {
    "plain": ({"mode": "plain"}, {}),
    "batched": ({"mode": "batched"}, {}),
    "ctas2": ({"mode": "batched", "ctas_per_sm": 2}, {}),
    "uninit": ({"mode": "batched", "check_uninit": True}, {"check_uninit": True}),
    "global": ({"mode": "plain", "check_global": True}, {"check_global": True}),
    "fused": ({"mode": "batched", "fused_check": True}, {}),
}
OPS = ["add", "sub", "mul", "and_", "or_", "xor", "shl", "shr", "min_", "max_", "slt", "sle", "seq", "sne"]


def random_kernel(seed: int, bdim: int, n: int, words: int) -> Asm:
    """r2 tid, r4 global id, r5..r8 values, r9 addresses and conditions, r10 loop counter."""
    G = rng.SplitMix64(seed)
    a = Asm()
    a.s2r(r2, TID).s2r(r3, BID).mul(r4, r3, bdim).add(r4, r4, r2).mul(r5, r4, 7).add(r5, r5, 1)
    val = R[5:9]

    def memory(kind):
        v = val[G.randint(0, 3)]
        if kind == 0:
            a.lds(v, r2, G.randint(0, 35))
        elif kind == 1:
            a.sts(r2, v, G.randint(0, 35))
        elif kind == 2:
            a.atoms(r2, v, G.randint(0, 3))
        elif kind == 3:                              # colliding stores, masked address
            a.and_(r9, v, 15).sts(r9, val[G.randint(0, 3)], G.randint(0, 2))
        elif kind == 4:                              # out of bounds for the highest tids
            a.lds(v, r2, words - max(1, bdim - 2))
        elif kind == 5:                              # an address read from memory
            a.lds(r9, r2).and_(r9, r9, 7).atoms(r9, v)
        elif kind == 6:
            a.ldg(v, r4)
        elif kind == 7:
            a.stg(r4, v, n)
        else:                                        # every fourth word, and below zero
            a.mul(r9, r2, 4).sts(r9, v, -8)

    def step(depth, i):
        what = G.randint(0, 13)
        if what == 0:
            for _ in range(G.randint(1, 9)):
                [lambda: a.mul(r5, r5, G.randint(-5, 9)), lambda: a.add(r5, r5, G.randint(-99, 99)),
                 lambda: a.sub(r5, r5, G.randint(0, 9)), lambda: a.shl(r5, r5, G.randint(0, 3))][G.randint(0, 3)]()
        elif what <= 2:
            for _ in range(G.randint(1, 5)):
                b = val[G.randint(0, 3)] if G.randint(0, 1) else G.randint(-3, 40)
                getattr(a, OPS[G.randint(0, len(OPS) - 1)])(val[G.randint(0, 3)], val[G.randint(0, 3)], b)
        elif what <= 6:
            memory(G.randint(0, 8))
        elif what == 7:
            d = [0, -1, 1, 7, -3][G.randint(0, 4)] if G.randint(0, 1) else val[G.randint(0, 3)]
            getattr(a, ["div", "rem"][G.randint(0, 1)])(val[G.randint(0, 3)], val[G.randint(0, 3)], d)
        elif what <= 10 and depth < 2:               # part by tid or by lane, join (at a barrier or not)
            skip = f"s{depth}_{i}_{a.pc}"
            if G.randint(0, 1):
                a.slt(r9, r2, G.randint(0, bdim)).brz(r9, skip)
            else:
                a.and_(r9, r2, [1, 3, 31, 32, 96][G.randint(0, 4)]).brnz(r9, skip)
            for j in range(G.randint(1, 3)):
                step(depth + 1, j)
            a.label(skip)
            if depth == 0 and G.randint(0, 1):
                a.bar()
        elif what == 11 and depth == 0:
            top = f"l{i}"
            a.mov(r10, G.randint(1, 4)).label(top)
            memory(G.randint(0, 3))
            a.add(r5, r5, 3).sub(r10, r10, 1).brnz(r10, top)
        elif depth == 0:
            [lambda: a.bar(), lambda: a.bar(), lambda: a.bar_count(val[G.randint(0, 3)], val[G.randint(0, 3)]),
             lambda: a.bar_or(val[G.randint(0, 3)], r9)][G.randint(0, 3)]()

    for i in range(14):
        step(0, i)
    if G.randint(0, 5) == 0:                         # some threads leave before a barrier: deadlock
        a.slt(r9, r2, G.randint(1, bdim)).brz(r9, "out").bar().label("out")
    return a.stg(r4, r5, 2 * n).exit()


def random_program(seed: int, bdim: int) -> Program:
    grid, words = 3, bdim + 40
    n = grid * bdim
    arena = np.zeros(3 * n, dtype=np.int32)
    arena[:n] = rng.uniform_mod(seed, n, 50)
    return Program(random_kernel(seed, bdim, n, words).assemble(), [0], [Launch(0, grid, bdim, words, (0, 0))], arena,
                   name=f"random_{seed}_{bdim}")


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1211_6193_gb300 import binding, build
    build.build()
    binding.load_library()
    return binding


def assert_same(B, progs, opts, oracle_kw):
    want = oracle.run(progs, **oracle_kw)
    got = B.check(progs, **opts)
    assert not np.any(got.status & (B.ST_LOG_OVERFLOW | B.ST_INTERNAL)), got.status
    for i, p in enumerate(progs):
        assert np.array_equal(got.arenas[i], want.arenas[i]), (i, p.name)
    assert list(got.status & 3) == list(want.status)
    assert got.report_tuples() == want.report_tuples()
    return got


@pytest.mark.parametrize("option", list(OPTIONS))
@pytest.mark.parametrize("bdim", BDIMS)
def test_random_kernels(B, bdim, option):
    opts, oracle_kw = OPTIONS[option]
    assert_same(B, [random_program(rng.derive(100 + bdim, i), bdim) for i in range(12)], opts, oracle_kw)


@pytest.mark.parametrize("blocks", [1, 7, 8, 9, 2047, 2048, 2049])
def test_report_compaction_sizes(B, blocks):
    """Racy blocks (every third one), over the sizes of the one-kernel compaction."""
    a = Asm().s2r(r2, TID).s2r(r3, BID).rem(r4, r3, 3).brnz(r4, "ok").and_(r11, r2, 3).sts(r11, r2).label("ok").exit()
    p = Program(a.assemble(), [0], [Launch(0, blocks, 32, 8, ())], np.zeros(4, np.int32))
    got = assert_same(B, [p], {"mode": "batched"}, {})
    assert len(got.reports) == 4 * ((blocks + 2) // 3)


def test_global_check_groups_by_program(B):
    """Racing programs with the same words, one without a launch among them, more runs than a tile."""
    def prog(i):
        a = Asm().s2r(r2, TID).s2r(r3, BID).mul(r4, r3, 64).add(r4, r4, r2).and_(r4, r4, 255).stg(r4, r2)
        a.ldg(r5, r4, i % 3).exit()
        return Program(a.assemble(), [0], [Launch(0, 9, 64, 1, ())] if i != 3 else [], np.zeros(300, np.int32))
    for mode in ("plain", "batched"):
        got = assert_same(B, [prog(i) for i in range(7)], {"mode": mode, "check_global": True}, {"check_global": True})
        assert len(got.reports) > 1500
    one = Asm().s2r(r2, BID).stg(r2, r2).exit()      # one record per word: no run
    wide = Program(one.assemble(), [0], [Launch(0, 3000, 1, 1, ())], np.zeros(3000, np.int32))
    assert len(assert_same(B, [wide], {"check_global": True}, {"check_global": True}).reports) == 0
    zero = Asm().s2r(r2, BID).mov(r3, 0).ldg(r4, r3).brnz(r2, "end").stg(r3, r2).label("end").exit()
    deep = Program(zero.assemble(), [0], [Launch(0, 3000, 1, 1, ())], np.zeros(4, np.int32))   # one long run
    assert len(assert_same(B, [deep], {"check_global": True}, {"check_global": True}).reports) == 1


@pytest.mark.parametrize("mode", ["plain", "batched"])
def test_global_check_run_lengths(B, mode):
    """Words used by one block to all of 1,400, the lengths around the run scan's limits (64 records, its
    tile of 1,024 and 256 behind it), odd words stored to, in launches that nothing orders too."""
    lengths = [1, 2, 3, 31, 62, 63, 64, 65, 66, 67, 127, 128, 129, 255, 256, 257, 258, 500, 640, 767, 768, 1000, 1022, 1023,
               1024, 1025, 1278, 1279, 1280, 1281, 1399, 1400]
    def prog(shift, unordered):
        a = Asm().s2r(r2, TID).s2r(r3, BID).ldg(r4, r2, 64).slt(r5, r3, r4).brz(r5, "end")
        a.and_(r9, r2, 1).brz(r9, "load").stg(r2, r3, 32).label("load").ldg(r10, r2, 32).label("end").exit()
        arena = np.zeros(96, np.int32)
        arena[64:] = np.roll(lengths, shift)
        launches = [Launch(0, 1400, 32, 1, (), stream=0)]
        if unordered:
            launches += [Launch(0, 1400, 32, 1, (), stream=1), Launch(0, 7, 32, 1, (), stream=2)]
        return Program(a.assemble(), [0], launches, arena, name=f"lengths_{shift}_{unordered}")
    progs = [prog(0, False), prog(5, True), prog(11, False)]
    want = oracle.run(progs, check_global=True)
    got = B.check(progs, mode=mode, check_global=True)
    assert not np.any(got.status)
    assert got.report_tuples() == want.report_tuples() and len(want.reports) > 60


def test_global_check_in_a_graph(B):
    """The sort's cooperative kernel under capture, and the graph run again."""
    progs = [random_program(rng.derive(7, i), 96) for i in range(6)]
    want = oracle.run(progs, check_global=True)
    with B.Context(mode="batched", check_global=True, use_graph=True) as ctx, ctx.load_programs(progs) as b:
        for _ in range(3):
            b.run_and_check()
            assert [tuple(int(x) for x in r) for r in b.fetch_reports()] == want.report_tuples()
