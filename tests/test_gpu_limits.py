"""Limits of a block at their exact edges: the round budget at every round of a kernel (what each
thread was doing when the rounds ran out, and how many instructions were executed), and an access
log that has been full for billions of accesses.  And the kernel form that carries most generated
batches, blocks of 129 to 512 threads with four simulated warps per warp, on random kernels."""
import numpy as np
import pytest

import oracle
from test_gpu_blocks import OPTIONS, B, assert_same, random_kernel, random_program  # noqa: F401 (the fixture)
from paper_1211_6193_gb300.workloads import rng
from paper_1211_6193_gb300.workloads.ir import TID, Asm, Launch, Program, r2, r3, r4, r5, r6, r7

pytestmark = pytest.mark.gpu


def assert_same_at(B, progs, budget, mode):
    want = oracle.run(progs, round_budget=budget)
    got = B.check(progs, mode=mode, round_budget=budget)
    assert got.report_tuples() == want.report_tuples(), budget
    assert list(got.status & 3) == list(want.status) and not np.any(got.status & B.ST_INTERNAL), budget
    assert got.stats.thread_instrs == want.thread_instrs, budget
    for i, p in enumerate(progs):
        assert np.array_equal(got.arenas[i], want.arenas[i]), (budget, p.name)


@pytest.mark.parametrize("mode", ["plain", "batched"])
@pytest.mark.parametrize("bdim", [33, 96, 128, 160, 512, 640, 1000])
def test_round_budget_at_a_parting_branch(B, bdim, mode):
    """Whole simulated warps go to a barrier or to the exit, the others go on; some part within."""
    progs = []
    for target in ("bar", "exit"):
        for split in (32, 48, 64, bdim - 1):
            for taken in (False, True):
                a = Asm().s2r(r2, TID).slt(r3, r2, split)
                (a.brnz if taken else a.brz)(r3, "t")
                a.add(r4, r4, 1).sts(r2, r4).add(r4, r4, 1).label("t")
                if target == "bar":
                    a.bar().add(r4, r4, 1)
                progs.append(Program(a.exit().assemble(), [0], [Launch(0, 2, bdim, bdim, ())], np.zeros(4, np.int32),
                                     name=f"{target}_{split}_{taken}"))
    for budget in range(1, 12):
        assert_same_at(B, progs, budget, mode)


def behind_large_block(p):
    """The program behind a launch of one block of 1024 threads that exits at once: in batched mode a
    program's launches run in one kernel form, that of its largest block (four simulated warps a warp)."""
    code = np.concatenate([p.code, Asm().exit().assemble()])
    return Program(code, [0, len(p.code)], [Launch(1, 1, 1024, 0, ())] + p.launches, p.global_init, name=p.name)


@pytest.mark.parametrize("four", [False, True])
@pytest.mark.parametrize("bdim", [64, 97, 128, 257, 512, 640, 1024])
def test_round_budget_at_every_round(B, bdim, four):
    grid, words = 2, bdim + 40
    n = grid * bdim
    progs = []
    for i in range(6):
        seed = rng.derive(900 + bdim, i)
        arena = np.zeros(3 * n, dtype=np.int32)
        arena[:n] = rng.uniform_mod(seed, n, 50)
        progs.append(Program(random_kernel(seed, bdim, n, words).assemble(), [0], [Launch(0, grid, bdim, words, (0, 0))],
                             arena, name=f"random_{i}"))
    longest = max(oracle.run([p]).rounds for p in progs)
    if four:
        progs = [behind_large_block(p) for p in progs]
    for budget in range(1, longest // grid + 2):
        assert_same_at(B, progs, budget, "plain" if budget & 1 and not four else "batched")


def test_full_log_stays_full(B):
    """A block whose log is full after four barrier intervals goes on for 2^32 more accesses, leaving
    the inner loop (a division by -1) between any two: its races are those of the first
    intervals, and the other program's results are untouched."""
    a = Asm().s2r(r2, TID).add(r3, r2, 1).and_(r3, r3, 1023).mov(r5, (1 << 18) + 64).mov(r7, -1)
    a.label("top").sts(r2, r5)
    for _ in range(16):
        a.lds(r4, r3).div(r6, r5, r7)
    a.bar().sub(r5, r5, 1).brnz(r5, "top").exit()
    long = Program(a.assemble(), [0], [Launch(0, 1, 1024, 1024, ())], np.zeros(4, np.int32), name="long")
    a = Asm().s2r(r2, TID).and_(r3, r2, 3).sts(r3, r2).exit()
    other = Program(a.assemble(), [0], [Launch(0, 5, 96, 8, ())], np.zeros(4, np.int32), name="other")
    got = B.check([long, other], mode="batched", round_budget=1 << 25, loop_log_records=1 << 16)
    assert got.status[0] == B.ST_LOG_OVERFLOW and got.status[1] == 0
    reports = got.report_tuples()
    mine = [r for r in reports if r[1] == 0]
    assert mine and {r[4] for r in mine} <= {0, 1, 2, 3}
    want = [(r[0], 1) + r[2:] for r in oracle.run([other]).report_tuples()]
    assert [r for r in reports if r[1] == 1] == want and want


@pytest.mark.parametrize("option", [o for o in OPTIONS if OPTIONS[o][0]["mode"] == "batched"])
@pytest.mark.parametrize("bdim", [129, 160, 255, 257, 384, 511, 512])
def test_four_simulated_warps_per_warp(B, bdim, option):
    opts, oracle_kw = OPTIONS[option]
    assert_same(B, [behind_large_block(random_program(rng.derive(700 + bdim, i), bdim)) for i in range(10)], opts, oracle_kw)


@pytest.mark.parametrize("option", ["plain", "global"])
@pytest.mark.parametrize("bdim", [129, 288, 512])
def test_four_simulated_warps_per_warp_in_large_grids(B, bdim, option):
    """Grids too large for the form of two simulated warps per warp (16 warps of it per SM)."""
    import torch
    opts, oracle_kw = OPTIONS[option]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    grid, words = 16 * sms // ((bdim + 63) // 64) + 1, bdim + 40
    n = grid * bdim
    progs = []
    for i in range(2):
        seed = rng.derive(800 + bdim, i)
        arena = np.zeros(3 * n, dtype=np.int32)
        arena[:n] = rng.uniform_mod(seed, n, 50)
        progs.append(Program(random_kernel(seed, bdim, n, words).assemble(), [0], [Launch(0, grid, bdim, words, (0, 0))],
                             arena, name=f"random_{i}"))
    assert_same(B, progs, opts, oracle_kw)
