"""Performance cases of the checker: what its users have it do, each through the public entry
points of ``paper_1211_6193_gb300.binding``.

A case names a workload (``kind``), its sizes and the context options.  Programs, launch shapes
and planted bugs follow from the case alone, the contents of the arenas from the seed.  A pass
is ``run_and_check`` on a loaded batch and then its results on the host: the reports, every
program's final arena and the status words, in page-locked memory as the serving loop fetches
them.  In the ``job`` kind a pass also loads the programs before and frees the batch after, as
a server does for every micro-batch.
"""
import ctypes

import numpy as np

from paper_1211_6193_gb300 import binding
from paper_1211_6193_gb300.workloads import families, fig1, ir, rng, stencil2d


def listed():
    return [
        # the paper's Figure 1 program: two launches of a few threads, the smallest check there is
        {"name": "fig1", "kind": "fig1", "mode": "plain"},
        # serving: one job of a few blocks arrives, is loaded, run, fetched and freed
        {"name": "job_1", "kind": "job", "mode": "batched", "programs": 1, "of": 512, "first": 3, "stream": 5},
        # serving under load: a micro-batch of jobs checked on a resident batch
        {"name": "micro_batch_16", "kind": "batch", "mode": "batched", "programs": 16, "of": 512, "first": 5, "stream": 5},
        # the batched workload: every sixteenth of the 4096 generated programs, grids 1..4096,
        # blocks of 32..1024 threads, all four families and planted bugs; the shapes the
        # autotuner picks for it
        {"name": "batch_256", "kind": "batch", "mode": "batched", "programs": 256, "of": 4096, "first": 0, "stream": 3,
         "ctas_per_sm": 2, "check_variant": 6},
        # the same kind of programs with the library's default shapes
        {"name": "batch_96_default", "kind": "batch", "mode": "batched", "programs": 96, "of": 4096, "first": 7,
         "stream": 3},
        # and one kernel launch per program launch
        {"name": "batch_64_plain", "kind": "batch", "mode": "plain", "programs": 64, "of": 4096, "first": 11, "stream": 3},
        # reads of unwritten shared words checked too
        {"name": "batch_64_uninit", "kind": "batch", "mode": "batched", "programs": 64, "of": 4096, "first": 19,
         "stream": 3, "check_uninit": True},
        # the plain single-program workload: tree reduction of 2^24 values, one missing barrier
        {"name": "reduction_2e24", "kind": "reduction", "mode": "plain", "blocks": 16384, "bdim": 1024, "omit": 3},
        # a reduction whose block is no multiple of a warp, race-free
        {"name": "reduction_ragged", "kind": "reduction", "mode": "plain", "blocks": 1501, "bdim": 333, "omit": -1},
        # global-memory race check on a reduction of 2^21 values
        {"name": "reduction_global", "kind": "reduction", "mode": "plain", "blocks": 2048, "bdim": 1024, "omit": 3,
         "check_global": True},
        # the log-heavy workload: 2-D stencil, 16 dependent launches, one without its barrier
        {"name": "stencil_2048", "kind": "stencil", "mode": "plain", "log2w": 11, "steps": 16, "buggy": 8},
        # a small grid iterated: the launches' dependences inside one persistent kernel, and the
        # paper's own method (access history kept by the interpreter)
        {"name": "stencil_256_fused", "kind": "stencil", "mode": "batched", "log2w": 8, "steps": 16, "buggy": 8,
         "fused_check": True},
    ]


def draw(rng_):
    """One more case: any kind, sizes log-uniform over the listed range, any mode and option."""
    def log_int(lo, hi):
        return int(round(lo * (hi / lo) ** rng_.random()))

    kind = rng_.choice(["job", "batch", "batch", "batch", "reduction", "reduction", "stencil"])
    case = {"kind": kind, "mode": rng_.choice(["plain", "batched"])}
    if kind in ("job", "batch"):
        n = log_int(1, 24 if kind == "job" else 128)
        case.update(programs=n, of=4096, first=rng_.randrange(4096 // n), stream=rng_.choice([3, 5]))
    elif kind == "reduction":
        bdim = rng_.choice([rng_.randint(1, 1024), 32 * rng_.randint(1, 32)])
        case.update(blocks=log_int(1, 4096), bdim=bdim, omit=rng_.randint(-1, families.reduction_levels(bdim) - 1))
    else:
        case.update(log2w=rng_.randint(6, 10), steps=rng_.randint(1, 16))
        case.update(buggy=rng_.randint(-1, case["steps"] - 1))
    option = rng_.choice([None, None, None, "check_uninit", "check_global", "fused_check", "ctas_per_sm"])
    if option == "ctas_per_sm":
        case.update(mode="batched", ctas_per_sm=2)
    elif option:
        case[option] = True
    return case


def _programs(case, seed):
    """The case's programs, their arenas filled from the seed."""
    kind = case["kind"]
    if kind == "fig1":
        p = fig1.program()
        arena = p.global_init.copy()
        arena[: fig1.N] = rng.uniform_mod(seed, fig1.N, 100)
        return [ir.Program(p.code, p.kernel_entry, p.launches, arena, p.name)]
    if kind == "reduction":
        return [families.reduction_plain(case["blocks"], case["bdim"], seed=rng.derive(seed, 0),
                                         omit_level=case["omit"] if case["omit"] >= 0 else None)]
    if kind == "stencil":
        return [stencil2d.program(case["log2w"], case["steps"], case["buggy"] if case["buggy"] >= 0 else None,
                                  seed=rng.derive(seed, 0))]
    step = case["of"] // case["programs"]
    return [families.build_family(families.draw_spec(rng.derive(case["stream"], i)), rng.derive(seed, i))
            for i in range(case["first"] % step, case["of"], step)[: case["programs"]]]


OPTIONS = ("ctas_per_sm", "check_variant", "check_uninit", "check_global", "fused_check")


class State:
    """A context, the programs, their batch (but for jobs) and the host buffer of the arenas."""

    def __init__(self, case, programs):
        self.programs = programs
        self.job = case["kind"] == "job"
        opts = {k: case[k] for k in OPTIONS if k in case}
        # device memory from the context's own pool for jobs, as the serving loop takes it
        self.ctx = binding.Context(mode=case["mode"], torch_allocator=not self.job, log_budget_mb=32 << 10, **opts)
        self.words = sum((p.global_init.size + 3) & ~3 for p in programs)
        self.arenas = binding.host_empty(self.words, np.int32, pinned=True)
        # room for the reports, kept from pass to pass (what no report fills stays zero)
        self.set_room(_report_room(case, programs))
        self.batch = None
        if self.job:                                     # inputs in page-locked receive buffers
            for p in programs:
                pinned = binding.host_empty(p.global_init.size, np.int32, pinned=True)
                pinned[:] = p.global_init
                p.global_init = pinned
        else:
            self.batch = self.ctx.load_programs(programs)

    def set_room(self, records):
        self.reports = binding.host_empty(records, binding.REPORT_DTYPE, pinned=True)
        self.reports.view(np.uint32)[:] = 0

    def __del__(self):
        if getattr(self, "batch", None) is not None:
            self.batch.free()
        if getattr(self, "ctx", None) is not None:
            self.ctx.close()


def _report_room(case, programs):
    """Records kept for the reports at first: a quarter of the threads of the launches that have
    a planted bug (reports come per racy word)."""
    bug = case.get("omit", -1) >= 0
    return _power_of_two(sum(l.grid * l.block_dim for p in programs for k, l in enumerate(p.launches)
                             if bug or p.meta.get("bug") or case.get("buggy", -1) == k) // 4)


def _power_of_two(n):
    return 1 << max(10, (n - 1).bit_length())


def prepare(case, seed):
    return State(case, _programs(case, seed))


def _fetch_reports(state, batch):
    """The reports into the kept buffer (grown when they do not fit); their number."""
    n = ctypes.c_uint64()
    while True:
        rc = state.ctx.lib.fetch_reports(state.ctx.handle, batch.handle, state.reports.ctypes.data,
                                         len(state.reports), ctypes.byref(n))
        if rc == binding.SR_OK:
            return n.value
        if rc != binding.SR_E_RANGE:
            raise binding.SimtCheckError(rc, state.ctx.lib.sr_last_error(state.ctx.handle).decode())
        state.set_room(_power_of_two(n.value))


def run(state):
    batch = state.ctx.load_programs(state.programs) if state.job else state.batch
    batch.run_and_check()
    n = _fetch_reports(state, batch)
    arenas = batch.fetch_memory(binding.SR_ALL_PROGRAMS, out=state.arenas)
    status = batch.all_status()
    if state.job:
        batch.free()
    return [n, state.reports.view(np.int32).reshape(-1, len(binding.REPORT_DTYPE)), arenas, status.view(np.int32)]


def exact(case, seed):
    return None                                          # whole numbers only


def _shortest_path(code, entry):
    """Fewest instructions a thread executes from `entry` to its exit."""
    ops, _, _, _, imms = ir.decode_fields(code)
    n = len(code)
    dist = {entry: 1}
    todo = [entry]
    while todo:                                          # breadth first
        nxt = []
        for pc in todo:
            op = int(ops[pc]) & 0x7F if pc < n else ir.EXIT
            if op == ir.EXIT:
                return dist[pc] if pc < n else dist[pc] - 1
            succ = [int(imms[pc])] if op in (ir.BRA, ir.BRZ, ir.BRNZ) else []
            if op != ir.BRA:
                succ.append(pc + 1)
            for s in succ:
                if s not in dist:
                    dist[s] = dist[pc] + 1
                    nxt.append(s)
        todo = nxt
    return 0


def work(case):
    """Bytes: every arena read and written once (for jobs across the host link; the reports,
    whose number follows from the planted bug, are left out).  Operations: the simulated
    thread-instructions on the shortest path through each kernel."""
    nbytes = flops = 0
    for p in _shapes(case):
        nbytes += 8 * p["words"] + 8 * len(p["code"])
        for kernel, threads in p["launches"]:
            flops += threads * _shortest_path(p["code"], p["entry"][kernel])
    return {"bytes": nbytes, "flops": flops}


def _shapes(case):
    """Code, launch sizes and arena words of the case's programs, without the arenas' contents."""
    kind = case["kind"]
    if kind == "reduction":
        b, t = case["blocks"], case["bdim"]
        code = families.reduction_kernel(t, case["omit"] if case["omit"] >= 0 else None).assemble()
        return [{"code": code, "entry": [0], "launches": [(0, b * t)], "words": b * t + b}]
    if kind == "stencil":
        w = 1 << case["log2w"]
        p = stencil2d.program(5, case["steps"], case["buggy"] if case["buggy"] >= 0 else None)
        code = stencil2d.stencil2d_kernel(case["log2w"]).assemble()
        return [{"code": code, "entry": [0, 0], "launches": [(l.kernel, w * w) for l in p.launches], "words": 2 * w * w}]
    if kind == "fig1":
        p = fig1.program()
        return [{"code": p.code, "entry": p.kernel_entry, "words": p.global_init.size,
                 "launches": [(l.kernel, l.grid * l.block_dim) for l in p.launches]}]
    out = []
    step = case["of"] // case["programs"]
    for i in range(case["first"] % step, case["of"], step)[: case["programs"]]:
        s = families.draw_spec(rng.derive(case["stream"], i))
        one = families.build_family(families.FamilySpec(**{**vars(s), "grid": 1}), 0)
        out.append({"code": one.code, "entry": [0], "launches": [(0, s.grid * s.bdim)],
                    "words": one.global_init.size * s.grid})
    return out
