// solo_loop.cuh - the interpreter's inner loop: the instructions of one warp's running set,
// executed one after the other until one needs the general steps of run_block (interp.cu).
//
// In PTX, because what bounds it is latency.  Shared memory and registers hold 20 to 30 warps per
// SM; a taken branch costs a warp some 24 cycles, an indexed jump 90 and an instruction in
// straight line 1 (timed in loops of them), and the same steps written in C++ executed two to four
// times the instructions (smsp__inst_executed).  Here:
//  - MOV, ADD and MUL with an immediate (SUB and SHL become them) are one multiply-add, and a
//    chain of them, each on the previous one's result, is a loop over its factors and addends
//    (set_runs lays them out); each group of the other operations is computed in straight line
//    under predicates;
//  - operand a of an instruction of a run is not read when it is the previous result (kept in
//    c), a result that the run overwrites is not written (set_runs), and a run's last round is
//    published when it starts (other warps wait on a clock for memory effects only);
//  - the next instruction is fetched ahead;
//  - the log's place for an access comes from an atomic whose result is used one access later:
//    the records of the last logged access stay in l/lw until the next logged access, or the
//    loop's end, writes them;
//  - a barrier that every thread of the block waits at, with nothing to report, is passed here,
//    with one CTA barrier: every warp reads all park entries and draws the same conclusion.
#pragma once
#include <cstddef>

#include "sr_internal.h"

namespace sr {
namespace {

// What the loop reads of the block (written at its start, kGroupConst): 16-byte groups.
struct SoloConst {
  uint32_t irs, rb, shs, sha;        // shared addresses of the code, the run lengths (8 bytes apart; less irs),
                                     // the shared array; its words
  unsigned long long arena;
  uint32_t arena_words, spin;
  uint32_t budget4, nrows, nthr, nw;  // (nrows, ncode: set and read in the debug build only)
  uint32_t tup, tps4;                // fused race check: the summaries, bytes per plane
  unsigned long long region;         // the log
  uint32_t wb, gcap, gblock, ncode;  // uninitialised-read check: the written words; global log: its size, the block
  unsigned long long gregion, pad2;  // the global log
};
static_assert(sizeof(SoloConst) == 96 && sizeof(SoloConst) <= kGroupBv - kGroupConst, "solo constants");
// Flags in: clocks are published (no other agent can run, or all others are at later rounds);
// several warps; log accesses; barriers may be passed here; the log is full; shared and global
// accesses may run here (or: with reads of unwritten words checked, with global accesses logged;
// then the fast bounds checks fail and the access takes the path behind them); every slot whose
// registers still matter is active; the active slots are slots 0..n-1 of every lane; no other agent
// can run; summaries instead of the log.  Flags out: the log is full; some threads wait at qw for
// the others to come there (kSoloAgents: some agents as a whole, at a barrier or exit); behind the
// CTA barrier of a simulated barrier that is not a plain release; a wait gave up.  (One register of
// bits instead of predicates: there are seven.)
enum : uint32_t {
  kSoloPub = 1, kSoloMany = 2, kSoloLog = 4, kSoloBar = 8, kSoloFull = 16, kSoloShared = 32, kSoloGlobal = 64, kSoloWhole = 128,
  kSoloRegular = 256, kSoloSolo = 512, kSoloFused = 1024, kSoloNested = 2048, kSoloAgents = 4096,
  kSoloToNest = 8192, kSoloToMerge = 16384,      // (inside: what follows the writing of kept records)
  kSoloAtBar = 32768, kSoloTimeout = 65536,
  kSoloUninit = 1 << 17, kSoloGlog = 1 << 18,    // (instead of kSoloShared, kSoloGlobal)
  kSoloBad = 1 << 19,                            // (debug build, out) an index check failed
  kSoloPending = 0x80000000u                     // (inside: records are kept)
};

// operands of the statement
#define Q_Q "%0"
#define Q_K4 "%1"
#define Q_GACC "%2"
#define Q_SACC "%3"
#define Q_EH "%4"
#define Q_NI "%5"
#define Q_FL "%6"
#define Q_QW "%7"
#define Q_MASK "%8"
#define Q_GB "%9"
#define Q_W "%10"
#define Q_RS "%11"
#define Q_STRIDE "%12"
#define Q_AM "%13"
#define Q_FCAP "%14"
#define Q_BUD "%15"
#define SR_STR2(x) #x
#define SR_STR(x) SR_STR2(x)

// Debug build: every index is checked before its access.  One that is out of range is noted in `bad`, and
// its access goes to an index in range (an operand's row, a place in the code) or is left out; the loop
// ends at the next instruction, with kSoloBad.
#if defined(SR_DEBUG_BOUNDS)
#define SR_ON(i) "@pg "
#define SR_D_DECL ".reg .pred px, pg;\n.reg .b32 bad, zrow, ncd, qlast, shr, awr, dx;\n"
#define SR_D_INIT                                                                                    \
  "mov.u32 bad, 0;\nld.shared.u32 zrow, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 36];\nsub.u32 zrow, zrow, 1;\n" \
  "ld.shared.u32 ncd, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 76];\nmad.lo.u32 qlast, ncd, 8, irs;\n" \
  "mov.u32 shr, sha;\nld.shared.u32 awr, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 24];\n"
#define SR_D_LIMIT(v, last) "setp.gt.u32 px, " v ", " last ";\n@px mov.u32 bad, 1;\n@px mov.u32 " v ", " last ";\n"
#define SR_D_ROW SR_D_LIMIT("ro", "zrow")        /* row of an operand */
#define SR_D_DST                                 /* row of a result that is written (ps) */             \
  "setp.gt.and.u32 px, ro, zrow, ps;\n@px mov.u32 bad, 1;\nsetp.le.and.u32 ps, ro, zrow, ps;\n"
#define SR_D_CODE(v) SR_D_LIMIT(v, "qlast")      /* address of an instruction */
#define SR_D_TARGET SR_D_LIMIT("y", "ncd")       /* pc of a branch's target */
#define SR_D_CHAIN SR_D_CODE("q") "@px mov.u32 t, 1;\n"
#define SR_D_SREG SR_D_LIMIT("y", "4")
#define SR_D_STOP "setp.ne.u32 px, bad, 0;\nvote.sync.any.pred px, px, 0xFFFFFFFF;\n@px bra.uni LDONE;\n"
#define SR_D_DONE "setp.ne.u32 px, bad, 0;\nvote.sync.any.pred px, px, 0xFFFFFFFF;\n@px or.b32 fl, fl, 0x80000;\n"
// pg: slot i is active and its index v below the limit
#define SR_D_BELOW(i, v, limit) "setp.lt.and.u32 pg, " v ", " limit ", s" #i ";\nxor.pred px, pg, s" #i ";\n@px mov.u32 bad, 1;\n"
#define SR_D_SH(i) SR_D_BELOW(i, "a" #i, "shr")
#define SR_D_GL(i) SR_D_BELOW(i, "a" #i, "awr")
#define SR_D_LOG(i) "add.u32 dx, base, lane;\nadd.u32 dx, dx, 32 * " #i ";\n" SR_D_BELOW(i, "dx", Q_FCAP)
// the written-words bitmap (pf: the lane changes the word at r1)
#define SR_D_WB                                                                                      \
  "add.u32 dx, shr, 31;\nshr.u32 dx, dx, 5;\nmad.lo.u32 dx, dx, 4, r0;\nsetp.ge.and.u32 px, r1, dx, pf;\n" \
  "@px mov.u32 bad, 1;\nsetp.lt.and.u32 px, r1, r0, pf;\n@px mov.u32 bad, 1;\n"                      \
  "setp.lt.and.u32 pf, r1, dx, pf;\nsetp.ge.and.u32 pf, r1, r0, pf;\n"
#else
#define SR_ON(i) "@s" #i " "
#define SR_D_DECL
#define SR_D_INIT
#define SR_D_ROW
#define SR_D_DST
#define SR_D_CODE(v)
#define SR_D_TARGET
#define SR_D_CHAIN
#define SR_D_SREG
#define SR_D_STOP
#define SR_D_DONE
#define SR_D_SH(i)
#define SR_D_GL(i)
#define SR_D_LOG(i)
#define SR_D_WB
#endif

// f for every slot
#define SR_E1(f) f(0)
#define SR_E2(f) f(0) f(1)
#define SR_E4(f) f(0) f(1) f(2) f(3)
// ALU groups (c: operand a and result, b: second operand)
#define SR_MAD(i) "mad.lo.u32 c" #i ", c" #i ", m, n;\n"
#define SR_MAD2(i) "mad.lo.u32 c" #i ", c" #i ", r0, r1;\n"
#define SR_MAD3(i) "mad.lo.u32 c" #i ", c" #i ", r2, r3;\n"
#define SR_MAD4(i) "mad.lo.u32 c" #i ", c" #i ", r4, r5;\n"
#define SR_REGOP(i) "@!pa mad.lo.u32 c" #i ", b" #i ", m, c" #i ";\n@pa mul.lo.u32 c" #i ", c" #i ", b" #i ";\n"
#define SR_SPLAT(i) "mov.u32 b" #i ", y;\n"
#define SR_LOGIC(i)                                                                          \
  "@pa and.b32 c" #i ", c" #i ", b" #i ";\n@pb xor.b32 c" #i ", c" #i ", b" #i ";\n"         \
  "@pc or.b32 c" #i ", c" #i ", b" #i ";\n"
#define SR_SHIFT(i)                                                                                   \
  "and.b32 t, b" #i ", 31;\n@pa shl.b32 c" #i ", c" #i ", t;\n@pb shr.s32 c" #i ", c" #i ", t;\n"     \
  "@pc min.s32 c" #i ", c" #i ", b" #i ";\n@pd max.s32 c" #i ", c" #i ", b" #i ";\n"
#define SR_COMPARE(i)                                                                        \
  "setp.lt.and.s32 pd, c" #i ", b" #i ", pa;\nsetp.eq.and.u32 pf, c" #i ", b" #i ", pb;\n"   \
  "or.pred pd, pd, pf;\nxor.pred pd, pd, pc;\nselp.u32 c" #i ", 1, 0, pd;\n"
// per slot of the set (s: active; a: addresses)
#define SR_SLOT(i) "and.b32 t, " Q_AM ", 1 << " #i ";\nsetp.ne.u32 s" #i ", t, 0;\n"
#define SR_KEEP0(i) "mov.u32 l" #i ", 0;\n"
#define SR_COUNT(i)                                                                          \
  "vote.sync.ballot.b32 t, s" #i ", 0xFFFFFFFF;\npopc.b32 t, t;\nadd.u32 n32, n32, t;\n"     \
  "@s" #i " add.u32 cnt, cnt, 1;\n"
// a branch that parts the threads (pz: BRZ): pc, some agent takes it as a whole; LNEST's new sets
#define SR_PARTS(i)                                                                          \
  "setp.eq.xor.u32 pf, a" #i ", 0, pz;\nand.pred pf, pf, s" #i ";\nvote.sync.any.pred pf, pf, 0xFFFFFFFF;\n" \
  "vote.sync.any.pred pd, s" #i ", 0xFFFFFFFF;\nnot.pred pf, pf;\nand.pred pf, pf, pd;\nor.pred pc, pc, pf;\n"
#define SR_NEST(i)                                                                           \
  "setp.eq.xor.u32 pf, a" #i ", 0, pz;\nnot.pred pd, pf;\nand.pred pd, pd, s" #i ";\n"       \
  "@pd or.b32 wm, wm, 1 << " #i ";\nand.pred s" #i ", s" #i ", pf;\n"
#define SR_JOIN(i) "and.b32 t, wm, 1 << " #i ";\nsetp.ne.or.u32 s" #i ", t, 0, s" #i ";\n"
#define SR_OUT(i) "@s" #i " or.b32 wm, wm, 1 << " #i ";\n"
#define SR_ADDR(i) "add.u32 a" #i ", a" #i ", y;\n"
#define SR_MAX(i) "@s" #i " max.u32 m, m, a" #i ";\n"
#define SR_MAXR(i) "@s" #i " max.u32 r0, r0, a" #i ";\n"
#define SR_LDSV(i) SR_D_SH(i) "mad.lo.u32 t, a" #i ", 4, shs;\n" SR_ON(i) "ld.shared.u32 c" #i ", [t];\n"
#define SR_LDGV(i) SR_D_GL(i) "mad.wide.u32 wide, a" #i ", 4, arena;\n" SR_ON(i) "ld.global.u32 c" #i ", [wide];\n"
#define SR_REDV(i) SR_D_SH(i) "mad.lo.u32 t, a" #i ", 4, shs;\n" SR_ON(i) "red.shared.add.u32 [t], b" #i ";\n"
#define SR_STSV(i) SR_D_SH(i) "mad.lo.u32 t, a" #i ", 4, shs;\n" SR_ON(i) "st.shared.u32 [t], b" #i ";\n"
#define SR_STGV(i) SR_D_GL(i) "mad.wide.u32 wide, a" #i ", 4, arena;\n" SR_ON(i) "st.global.u32 [wide], b" #i ";\n"
#define SR_SREG(i) "add.u32 m, u, 32 * " #i ";\nselp.b32 c" #i ", m, t, pa;\n"
#define SR_ZERO(i) "mov.u32 c" #i ", 0;\n"
#define SR_OFF(i) "add.u32 u, m, 32 * " #i ";\nxor.b32 u, u, a" #i ";\n@s" #i " or.b32 n, n, u;\n"
// stores that are consecutive within each slot only: pc, some slot's are not; lowest and highest address
#define SR_OFF1(i)                                                                           \
  "vote.sync.ballot.b32 t, s" #i ", 0xFFFFFFFF;\nbrev.b32 t, t;\nclz.b32 t, t;\nmin.u32 t, t, 31;\n" \
  "shfl.sync.idx.b32 u, a" #i ", t, 31, 0xFFFFFFFF;\nsub.u32 u, u, t;\nadd.u32 u, u, lane;\n" \
  "setp.ne.and.u32 pf, u, a" #i ", s" #i ";\nor.pred pc, pc, pf;\n@s" #i " min.s32 need, need, a" #i ";\n" \
  "@s" #i " max.s32 qend, qend, a" #i ";\n"
#define SR_STSO(i) SR_STSV(i) "bar.warp.sync 0xFFFFFFFF;\n"
#define SR_STGO(i) SR_STGV(i) "bar.warp.sync 0xFFFFFFFF;\n"
#define SR_DIVV(i) "div.s32 c" #i ", a" #i ", y;\n"
#define SR_REMV(i) "rem.s32 c" #i ", a" #i ", y;\n"
#define SR_DIVOK(i) "add.u32 t, b" #i ", 1;\nsetp.le.and.u32 pf, t, 1, s" #i ";\nor.pred pc, pc, pf;\n"
#define SR_DIVRV(i) "div.s32 c" #i ", a" #i ", b" #i ";\n"
#define SR_REMRV(i) "rem.s32 c" #i ", a" #i ", b" #i ";\n"
// 45 DIV, 47 REM by registers that are neither 0 nor -1 in any active thread
#define SR_NO_DIVR(E, LDB) "bra.uni LEND;\n"
#define SR_DIVR(E, LDB)                                                                              \
  "setp.eq.u32 pa, u, 45;\nsetp.eq.or.u32 pf, u, 47, pa;\n@!pf bra.uni LEND;\nprmt.b32 ro, x, 0, 0x4443;\n"   \
  SR_D_ROW "mad.lo.u32 ro, ro, " Q_STRIDE ", " Q_RS ";\n" LDB "setp.ne.u32 pc, 0, 0;\n" E(SR_DIVOK)    \
  "vote.sync.any.pred pc, pc, 0xFFFFFFFF;\n@pc bra.uni LEND;\n@!pa bra.uni LREMR;\n" E(SR_DIVRV)      \
  "bra.uni LDIV1;\nLREMR:\n" E(SR_REMRV) "bra.uni LDIV1;\n"
#define SR_BITS(i) "@s" #i " or.b32 m, m, a" #i ";\n@s" #i " min.u32 n, n, a" #i ";\n"
#define SR_KEEP(i) "mov.u32 l" #i ", a" #i ";\n"
#define SR_REC(i)                                                                                    \
  SR_D_LOG(i)                                                                                        \
  "shl.b32 t, l" #i ", 24;\nadd.u32 t, t, lw;\nadd.u32 lw, lw, 0x80000;\nshr.u32 u, l" #i ", 8;\n"   \
  "or.b32 u, u, eh;\n" SR_ON(i) "st.global.v2.u32 [wide + 256 * " #i "], {t, u};\n"
#define SR_REC_ANY(i) /* any set of threads, and a log that may be full */                           \
  "vote.sync.ballot.b32 t, s" #i ", 0xFFFFFFFF;\nand.b32 u, t, r0;\npopc.b32 u, u;\nadd.u32 u, u, m;\n" \
  "popc.b32 t, t;\nadd.u32 m, m, t;\nsetp.lt.and.u32 pf, u, " Q_FCAP ", s" #i ";\n"                  \
  "setp.lt.and.u32 pf, base, " Q_FCAP ", pf;\nmad.wide.u32 wide, u, 8, region;\n"              \
  "shl.b32 r1, l" #i ", 24;\nadd.u32 r1, r1, lw;\nadd.u32 lw, lw, 0x80000;\nshr.u32 r2, l" #i ", 8;\n" \
  "or.b32 r2, r2, eh;\n@pf st.global.v2.u32 [wide], {r1, r2};\n"
#define SR_PUT(i) "@s" #i " st.shared.u32 [ro + 4 * " #i "], c" #i ";\n"
// uninitialised-read check (r0: the bitmap of written words): pa, an active thread reads an unwritten
// word; the words of a store (consecutive within a slot), of an atomic
#define SR_WBR(i)                                                                                    \
  SR_D_SH(i)                                                                                         \
  "shr.u32 t, a" #i ", 5;\nmad.lo.u32 t, t, 4, r0;\nand.b32 u, a" #i ", 31;\nmov.u32 n, 0xFFFFFFFF;\n" \
  SR_ON(i) "ld.shared.u32 n, [t];\nshr.u32 n, n, u;\nand.b32 n, n, 1;\nsetp.eq.or.u32 pa, n, 0, pa;\n"
#define SR_WBS(i)                                                                                    \
  "vote.sync.ballot.b32 t, s" #i ", 0xFFFFFFFF;\nbrev.b32 u, t;\nclz.b32 u, u;\nmin.u32 u, u, 31;\n"  \
  "shfl.sync.idx.b32 r1, a" #i ", u, 31, 0xFFFFFFFF;\nsub.u32 r1, r1, u;\nand.b32 u, r1, 31;\n"       \
  "shl.b32 r2, t, u;\nsub.u32 u, 32, u;\nshr.u32 r3, t, u;\nshr.s32 r1, r1, 5;\nsetp.eq.u32 pa, lane, 1;\n" \
  "@pa mov.u32 r2, r3;\nadd.u32 r1, r1, lane;\nmad.lo.u32 r1, r1, 4, r0;\nsetp.lt.u32 pf, lane, 2;\n" \
  "setp.ne.and.u32 pf, r2, 0, pf;\n" SR_D_WB "@pf red.shared.or.b32 [r1], r2;\n"
#define SR_WBA(i)                                                                                    \
  SR_D_SH(i)                                                                                         \
  "shr.u32 t, a" #i ", 5;\nmad.lo.u32 t, t, 4, r0;\nand.b32 u, a" #i ", 31;\nmov.u32 r1, 1;\n"        \
  "shl.b32 r1, r1, u;\n" SR_ON(i) "red.shared.or.b32 [t], r1;\n"
// the access's records in the global log (as log_global), kind << 12
#define SR_GREC(i)                                                                                   \
  "vote.sync.ballot.b32 t, s" #i ", 0xFFFFFFFF;\nand.b32 u, t, r0;\npopc.b32 u, u;\nadd.u32 u, u, m;\n" \
  "popc.b32 t, t;\nadd.u32 m, m, t;\nsetp.lt.and.u32 pf, u, r1, s" #i ";\nsetp.lt.and.u32 pf, r5, r1, pf;\n" \
  "mad.wide.u32 wide, u, 16, region;\n@pf st.global.v4.u32 [wide], {a" #i ", r4, r3, r2};\nadd.u32 r3, r3, 0x200000;\n"
#define SR_GLOG(E, kind)                                                                             \
  "ld.shared.v4.u32 {r0, r1, r2, r3}, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 64];\n"                \
  "ld.shared.u64 region, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 80];\n"                             \
  "ld.shared.u32 r5, [" Q_GB " + " SR_STR(SR_GROUP_BV) " + 44];\nsetp.eq.u32 pf, lane, 0;\n"         \
  "setp.lt.and.u32 pf, r5, r1, pf;\n@pf atom.shared.add.u32 r5, [" Q_GB " + " SR_STR(SR_GROUP_BV) " + 44], n32;\n" \
  "sub.u32 r3, q, irs;\nshr.u32 r3, r3, 3;\nmad.lo.u32 r3, tid0, 65536, r3;\nadd.u32 r3, r3, " #kind " << 12;\n" \
  "shr.u32 r4, eh, 6;\nmov.u32 r0, %%lanemask_lt;\nshfl.sync.idx.b32 r5, r5, 0, 31, 0xFFFFFFFF;\nmov.u32 m, r5;\n" \
  E(SR_GREC) "sub.u32 t, r1, r5;\nsetp.lt.u32 pf, t, n32;\nsetp.ge.or.u32 pf, r5, r1, pf;\n"        \
  "setp.eq.and.u32 pf, lane, 0, pf;\nmov.u32 t, 1;\n@pf atom.shared.or.b32 t, [" Q_GB " + " SR_STR(SR_GROUP_BV) " + 20], t;\n"
// fused race check: the access of slot i into its word's summary (tuple_add), pc in r0, tid r1 (of
// slot 0); the returned values (in b) are used when every slot's atomics are under way
#define SR_TUPLE(i, k2)                                                                              \
  SR_D_SH(i) "mad.lo.u32 t, a" #i ", 4, tup;\nmad.lo.u32 u, tps4, 6, t;\n" SR_ON(i) "red.shared.min.u32 [u], r0;\n" \
  "add.u32 u, u, tps4;\n" SR_ON(i) "red.shared.max.u32 [u], r0;\nmad.lo.u32 u, tps4, " #k2 ", t;\n"  \
  "add.u32 b" #i ", r1, 32 * " #i ";\n" SR_ON(i) "atom.shared.min.u32 b" #i ", [u], b" #i ";\n"
#define SR_TUPLE_OLD(i, k21)                                                                         \
  "add.u32 r2, r1, 32 * " #i ";\nsetp.ne.and.u32 pf, b" #i ", r2, s" #i ";\n"                       \
  "setp.ne.and.u32 pf, b" #i ", 0xFFFFFFFF, pf;\nmax.u32 t, b" #i ", r2;\n"                         \
  "mad.lo.u32 u, a" #i ", 4, tup;\nmad.lo.u32 u, tps4, " #k21 ", u;\n@pf red.shared.min.u32 [u], t;\n"
#define SR_TUPLE0(i) SR_TUPLE(i, 0)
#define SR_TUPLE1(i) SR_TUPLE(i, 2)
#define SR_TUPLE2(i) SR_TUPLE(i, 4)
#define SR_TUPLE_OLD0(i) SR_TUPLE_OLD(i, 1)
#define SR_TUPLE_OLD1(i) SR_TUPLE_OLD(i, 3)
#define SR_TUPLE_OLD2(i) SR_TUPLE_OLD(i, 5)
#define SR_NO_TUP(E, kind)
#define SR_TUP(E, kind)                                                                              \
  "and.b32 t, fl, 1024;\nsetp.eq.u32 pf, t, 0;\n@pf bra.uni LNOTUP" #kind ";\n" \
  "sub.u32 r0, q, irs;\nshr.u32 r0, r0, 3;\nmov.u32 r1, tid0;\n" \
  "ld.shared.v2.u32 {tup, tps4}, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 48];\n" E(SR_TUPLE##kind) E(SR_TUPLE_OLD##kind) "add.u32 sacc, sacc, cnt;\nLNOTUP" #kind ":\n"
// end of an instruction of a run (q already past it): the result's store, and the next
// instruction or the run's end
#define SR_TAIL(STC, more)                                                                           \
  "setp.ge.u32 pe, q, qend;\nand.b32 t, x, 128;\nsetp.eq.or.u32 ps, t, 0, pe;\n"                     \
  "prmt.b32 ro, x, 0, 0x4441;\nsetp.ne.and.u32 ps, ro, 31, ps;\n" SR_D_DST "mad.lo.u32 ro, ro, " Q_STRIDE ", " Q_RS ";\n" \
  "@!pw bra.uni LPART;\n@ps " STC "mov.u32 x, nx;\nmov.u32 y, ny;\nmov.u32 keep, 64;\n"              \
  "@!pe bra.uni LALU;\n" more
// end of a memory or control instruction
#define SR_FIN                                                                                       \
  "add.u32 q, q, 8;\nadd.u32 k4, k4, 4;\nmov.u32 x, nx;\nmov.u32 y, ny;\nbar.warp.sync 0xFFFFFFFF;\n" \
  "@pp st.release.cta.shared.u32 [myclk], k4;\nsetp.lt.u32 pe, k4, bud;\nsetp.lt.and.u32 pe, q, qw, pe;\n" \
  "@pe bra.uni LTOP;\nbra.uni LSTOP;\n"
// row d from c (a memory instruction's result)
#define SR_ROW(STC, part, back)                                                                      \
  "prmt.b32 ro, x, 0, 0x4441;\nsetp.ne.u32 ps, ro, 31;\n" SR_D_DST "mad.lo.u32 ro, ro, " Q_STRIDE ", " Q_RS ";\n" \
  "@!pw bra.uni " part ";\n@ps " STC back ":\n"
// reserve the log's place for this access and keep its records to be written later
#define SR_LOG(E, kind)                                                                              \
  E(SR_KEEP) "and.b32 t, fl, 4;\nmov.u32 base, 0xFFFFFFFF;\nsetp.lt.u32 pf, lane, t;\nsetp.eq.and.u32 pf, lane, 0, pf;\n" \
  "@pf atom.shared.add.u32 base, [" Q_GB " + " SR_STR(SR_GROUP_BV) " + 16], n32;\n"                  \
  "sub.u32 lw, q, irs;\nshr.u32 lw, lw, 3;\nmad.lo.u32 lw, tid0, 16384, lw;\nadd.u32 lw, lw, " #kind " << 12;\n" \
  "and.b32 t, fl, 20;\nsetp.ne.u32 pf, t, 0;\n@pf or.b32 fl, fl, 0x80000000;\n"
// write the records kept by SR_LOG (coalesced at once when the set is regular and they fit)
#define SR_FLUSH(E, tag)                                                                             \
  "shfl.sync.idx.b32 base, base, 0, 31, 0xFFFFFFFF;\nld.shared.u64 region, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 56];\n" \
  "and.b32 fl, fl, 0x7FFFFFFF;\nand.b32 t, fl, 2304;\nsetp.eq.u32 pf, t, 256;\n"                     \
  "sub.u32 t, " Q_FCAP ", base;\nsetp.ge.u32 pa, t, n32;\nsetp.lt.and.u32 pa, base, " Q_FCAP ", pa;\n" \
  "and.pred pf, pf, pa;\nadd.u32 t, base, lane;\nmad.wide.u32 wide, t, 8, region;\n@!pf bra.uni LANY" tag ";\n" E(SR_REC) \
  "LFLUSHED" tag ":\n"
#define SR_FLUSH_ANY(E, tag)                                                                         \
  "LANY" tag ":\nmov.u32 m, base;\nmov.u32 r0, %%lanemask_lt;\n" E(SR_REC_ANY)                       \
  "@pa bra.uni LFLUSHED" tag ";\nand.b32 t, fl, 4;\nsetp.ne.u32 pf, t, 0;\nsetp.eq.and.u32 pf, lane, 0, pf;\n" \
  "mov.u32 t, 1;\n@pf atom.shared.or.b32 t, [" Q_GB " + " SR_STR(SR_GROUP_BV) " + 20], t;\n"          \
  "and.b32 fl, fl, 0xFFFFFFFB;\nor.b32 fl, fl, 16;\nbra.uni LFLUSHED" tag ";\n"
// wait (bounded) until every other warp's clock has reached `need` (of this interval's parity: a
// warp still parked at the last barrier shows the other parity and reads as lower; the lanes that
// stand for no other warp read the warp's own clock, which is at `need` already)
#define SR_POLL(tag)                                                                                 \
  "mov.u32 n, 0;\n"                                                                                  \
  "LPOLL" tag ":\nld.acquire.cta.shared.u32 clk, [clks];\nsub.u32 clk, clk, need;\n"                 \
  "setp.ge.s32 pf, clk, 0;\n"                                                                         \
  "vote.sync.all.pred pf, pf, 0xFFFFFFFF;\n@pf bra.uni LPOLLED" tag ";\n"                            \
  "add.u32 n, n, 1;\nld.shared.u32 u, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 28];\nsetp.ge.u32 pf, n, u;\n@pf bra.uni LTIMEOUT;\n"                              \
  "setp.gt.u32 pf, n, 32;\n@pf nanosleep.u32 32;\nbra.uni LPOLL" tag ";\nLPOLLED" tag ":\n"
// pf: the highest address v is below the array's real size (word `at` of the constants), and the
// access may run here in its second form (flag)
#define SR_REAL(flag, v, at)                                                                         \
  "and.b32 t, fl, " flag ";\nsetp.ne.u32 pf, t, 0;\nld.shared.u32 t, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + " at "];\n" \
  "setp.lt.and.u32 pf, " v ", t, pf;\nvote.sync.all.pred pf, pf, 0xFFFFFFFF;\n"
#define SR_SOLO_ASM(V, REGS, LDC, LDB, STC, LDA, E, TUP, DIVR)                                                            \
  asm volatile(                                                                                                     \
      "{\n"                                                                                                         \
      ".reg .pred pa, pb, pc, pd, pe, pf, ps, pw, pp, pm, pz, s0, s1, s2, s3;\n"                                    \
      ".reg .b32 x, y, nx, ny, m, n, t, u, ro, keep, q, qend, k4, base, lw, eh, n32, clk, need, lane, tid0;\n"      \
      ".reg .b32 gacc, sacc, cnt, r0, r1, r2, r3, r4, r5, irs, shs, sha, awords, bud, tup, tps4, clks, myclk;\n"    \
      SR_D_DECL ".reg .b32 ni, kst, qw, wm, fl;\n.reg .b64 wide, arena, region;\n.reg .b32 " REGS ";\n"                      \
      "ld.shared.v4.u32 {irs, t, shs, sha}, [" Q_GB " + " SR_STR(SR_GROUP_CONST) "];\n"                             \
      "ld.shared.u32 t, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 44];\n"                                            \
      SR_D_INIT "mov.u32 q, " Q_Q ";\n" SR_D_CODE("q") "mov.u32 bud, " Q_BUD ";\nld.shared.v2.u32 {x, y}, [q];\n"                \
      "mov.u32 k4, " Q_K4 ";\nmov.u32 eh, " Q_EH ";\nmov.u32 fl, " Q_FL ";\nmov.u32 qw, " Q_QW ";\nmov.u32 wm, 0;\n"  \
      "mov.u32 lane, %%laneid;\nmov.u32 gacc, " Q_GACC ";\nmov.u32 sacc, " Q_SACC ";\nmov.u32 ni, " Q_NI ";\n"        \
      "and.b32 kst, k4, 0x7FFFFFFF;\nmad.lo.u32 tid0, " Q_W ", 32 * " #V ", lane;\n"                                \
      "mad.lo.u32 myclk, " Q_W ", 4, " Q_GB ";\nmad.lo.u32 clks, lane, 4, " Q_GB ";\n"                              \
      "setp.ge.u32 pf, lane, t;\n@pf mov.u32 clks, myclk;\n"      \
      "and.b32 t, fl, 32;\nsetp.eq.u32 pf, t, 0;\n@pf mov.u32 sha, 0;\n" /* (no shared access is in bounds) */     \
      "and.b32 t, fl, 1;\nsetp.ne.u32 pp, t, 0;\nsetp.eq.and.u32 pp, lane, 0, pp;\n"                              \
      "mov.u32 base, 0;\nmov.u32 lw, 0;\n" E(SR_KEEP0) E(SR_SLOT)                                                  \
      "and.b32 t, fl, 128;\nsetp.ne.u32 pw, t, 0;\n@pp st.release.cta.shared.u32 [myclk], k4;\n"                    \
      "bar.warp.sync 0xFFFFFFFF;\n"                                                                                \
      "LMASK:\n" /* the set has changed: its numbers */                                                             \
      "mov.u32 n32, 0;\nmov.u32 cnt, 0;\n" E(SR_COUNT)                                                             \
      "setp.lt.u32 pe, k4, bud;\nsetp.lt.and.u32 pe, q, qw, pe;\n@!pe bra.uni LSTOP;\n"                             \
      "LTOP:\n" SR_D_CODE("q") SR_D_STOP                                                                                                     \
      "and.b32 u, x, 63;\nsetp.ge.u32 pm, u, 32;\n@pm bra.uni LMEM;\n" /* a run starts */                           \
      "ld.shared.u32 u, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 4];\nadd.u32 t, q, u;\nld.shared.u8 t, [t];\n"                           \
      "sub.u32 u, bud, k4;\nshr.u32 u, u, 2;\nand.b32 r0, fl, 513;\nsetp.eq.u32 pf, r0, 1;\n@pf mov.u32 u, 255;\n"   \
      "min.u32 t, t, u;\nsub.u32 u, qw, q;\nshr.u32 u, u, 3;\n" /* (up to other agents' round: not cut, see bud) */  \
      "min.u32 t, t, u;\nmad.lo.u32 qend, t, 8, q;\n" SR_D_CODE("qend") "mad.lo.u32 k4, t, 4, k4;\n"                                     \
      "min.u32 r0, k4, bud;\n@pp st.release.cta.shared.u32 [myclk], r0;\nmov.u32 keep, 0;\n"                                              \
      "LALU:\n"                                                                                                     \
      "and.b32 t, x, keep;\nsetp.eq.u32 pf, t, 0;\n"                                                                \
      "prmt.b32 ro, x, 0, 0x4442;\n" SR_D_ROW "mad.lo.u32 ro, ro, " Q_STRIDE ", " Q_RS ";\n@pf " LDC                            \
      "and.b32 u, x, 63;\nsetp.gt.u32 pf, u, 2;\n@pf bra.uni LGEN;\n"                                               \
      /* 0 MOV, 1 ADD, 2 MUL with an immediate: c * m + n, for t instructions in a row */                           \
      "prmt.b32 t, x, 0, 0x4443;\nmad.lo.u32 q, t, 8, q;\n" SR_D_CHAIN "ld.shared.v2.u32 {nx, ny}, [q];\n"                        \
      "setp.eq.u32 pf, u, 2;\nselp.u32 m, y, u, pf;\nselp.u32 n, 0, y, pf;\n" E(SR_MAD)                             \
      "setp.gt.u32 pf, t, 1;\n@pf bra.uni LCHAIN;\nLCHAINED:\n" SR_TAIL(STC, "")                                    \
      "LRUNEND:\nmov.u32 q, qend;\n" /* (cut by its largest length, the rounds left or the lowest waiting pc) */    \
      "setp.lt.u32 pe, k4, bud;\nsetp.lt.and.u32 pe, q, qw, pe;\n@!pe bra.uni LSTOP;\n"                        \
      "and.b32 u, x, 63;\nsetp.lt.u32 pf, u, 32;\n@pf bra.uni LTOP;\n"                                              \
      "LMEM:\n" /* memory and control: u = the form */                                                              \
      "ld.shared.v2.u32 {nx, ny}, [q + 8];\nprmt.b32 ro, x, 0, 0x4442;\n" SR_D_ROW "mad.lo.u32 ro, ro, " Q_STRIDE ", " Q_RS ";\n" LDA \
      "setp.ge.u32 pf, u, 34;\n@pf bra.uni LMORE;\nld.acquire.cta.shared.u32 clk, [clks];\nmov.u32 qend, u;\n"      \
      "setp.ge.s32 pf, fl, 0;\n@pf bra.uni LMEM1;\n" SR_FLUSH(E, "A")                                                                      \
      "LMEM1:\n" E(SR_ADDR) "setp.eq.u32 pf, qend, 33;\n@pf bra.uni LSTS;\n"                                        \
      /* 32 LDS */                                                                                                  \
      "mov.u32 m, 0;\nsub.u32 clk, clk, k4;\n" E(SR_MAX)                                                            \
      "setp.lt.u32 pf, m, sha;\nsetp.ge.and.s32 pa, clk, 0, pf;\n"    \
      "vote.sync.all.pred pa, pa, 0xFFFFFFFF;\n"                                                                    \
      "@!pa bra.uni LLDSW;\nLLDSW1:\nbar.warp.sync 0xFFFFFFFF;\n" E(SR_ZERO) E(SR_LDSV) SR_LOG(E, 0) TUP(E, 0)      \
      SR_ROW(STC, "LROWA", "LROWA1") SR_FIN                                                                         \
      "LLDSW:\nvote.sync.all.pred pf, pf, 0xFFFFFFFF;\n@!pf bra.uni LLDSU;\n"                                       \
      "mov.u32 need, k4;\n" SR_POLL("A") "bra.uni LLDSW1;\n"                                                       \
      "LLDSU:\n" SR_REAL("131072", "m", "12") "@!pf bra.uni LEND;\nmov.u32 need, k4;\n" SR_POLL("D")               \
      "ld.shared.u32 r0, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 64];\nsetp.ne.u32 pa, 0, 0;\n"                    \
      "bar.warp.sync 0xFFFFFFFF;\n" E(SR_WBR) "vote.sync.any.pred pa, pa, 0xFFFFFFFF;\n@pa bra.uni LEND;\n"         \
      "bra.uni LLDSW1;\n"                                                        \
      /* 33 STS: consecutive words, one per thread, cannot collide */                                               \
      "LSTS:\n"                                                                                                     \
      "prmt.b32 ro, x, 0, 0x4443;\n" SR_D_ROW "mad.lo.u32 ro, ro, " Q_STRIDE ", " Q_RS ";\n" LDB                                \
      "vote.sync.ballot.b32 t, s0, 0xFFFFFFFF;\nsetp.ne.u32 pa, t, 0;\nbrev.b32 t, t;\nclz.b32 t, t;\nmin.u32 t, t, 31;\n" \
      "shfl.sync.idx.b32 need, a0, t, 31, 0xFFFFFFFF;\nsub.u32 need, need, t;\nadd.u32 m, need, lane;\n"      \
      "mov.u32 n, 0;\nmov.u32 r0, 0;\n" E(SR_OFF) E(SR_MAXR)                                                        \
      "setp.eq.and.u32 pf, n, 0, pa;\nsetp.lt.and.u32 pf, r0, sha, pf;\n"                   \
      "vote.sync.all.pred pf, pf, 0xFFFFFFFF;\n@!pf bra.uni LSTSX;\nmov.u32 m, 1;\nand.b32 t, fl, 2;\nsetp.ne.u32 pf, t, 0;\nmov.u32 r5, 0;\n@pf bra.uni LRANGE;\n" \
      "LSTS1:\n" E(SR_STSV) "LSTS2:\n" SR_LOG(E, 1) TUP(E, 1) SR_FIN                                                           \
      /* 34 BRZ, 35 BRNZ */                                                                                         \
      "LMORE:\nsetp.ge.u32 pf, u, 36;\n@pf bra.uni LMORE2;\nmov.u32 m, 0;\nmov.u32 n, 0xFFFFFFFF;\n" E(SR_BITS)     \
      "setp.eq.u32 pa, m, 0;\nsetp.ne.u32 pb, n, 0;\nvote.sync.all.pred pa, pa, 0xFFFFFFFF;\n"                      \
      "vote.sync.all.pred pb, pb, 0xFFFFFFFF;\nor.pred pf, pa, pb;\n@!pf bra.uni LPARTS;\n" /* both ways */           \
      "setp.eq.xor.u32 pf, u, 34, pb;\n@pf bra.uni LTAKE;\n" SR_FIN                                                 \
      "LTAKE:\n" SR_D_TARGET "mad.lo.u32 q, y, 8, irs;\nld.shared.v2.u32 {nx, ny}, [q];\nsub.u32 q, q, 8;\n" SR_FIN                \
      /* 36 LDG, 37 STG */                                                                                          \
      "LMORE2:\nld.shared.u64 arena, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 16];\n"                                \
      "ld.shared.u32 awords, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 24];\nand.b32 t, fl, 64;\nsetp.eq.u32 pf, t, 0;\n@pf mov.u32 awords, 0;\n"                           \
      "ld.acquire.cta.shared.u32 clk, [clks];\nsetp.ge.u32 pf, u, 38;\n@pf bra.uni LMORE3;\n" E(SR_ADDR)   \
      "setp.eq.u32 pf, u, 37;\n@pf bra.uni LSTG;\nmov.u32 m, 0;\nsub.u32 clk, clk, k4;\n" E(SR_MAX)                 \
      "setp.lt.u32 pf, m, awords;\nsetp.ge.and.s32 pa, clk, 0, pf;\n" \
      "vote.sync.all.pred pa, pa, 0xFFFFFFFF;\n"                                                                    \
      "@!pa bra.uni LLDGW;\nLLDGW1:\nbar.warp.sync 0xFFFFFFFF;\n" E(SR_ZERO) E(SR_LDGV)                             \
      "add.u32 gacc, gacc, cnt;\n" SR_ROW(STC, "LROWB", "LROWB1") SR_FIN                                            \
      "LLDGW:\nvote.sync.all.pred pf, pf, 0xFFFFFFFF;\n@!pf bra.uni LLDGU;\n"                                       \
      "mov.u32 need, k4;\n" SR_POLL("B") "bra.uni LLDGW1;\n"                                                       \
      "LLDGU:\n" SR_REAL("262144", "m", "24") "@!pf bra.uni LEND;\nmov.u32 need, k4;\n" SR_POLL("E")               \
      SR_GLOG(E, 0) "bra.uni LLDGW1;\n"                                                        \
      "LSTG:\n"                                                                                                     \
      "prmt.b32 ro, x, 0, 0x4443;\n" SR_D_ROW "mad.lo.u32 ro, ro, " Q_STRIDE ", " Q_RS ";\n" LDB                                \
      "vote.sync.ballot.b32 t, s0, 0xFFFFFFFF;\nsetp.ne.u32 pa, t, 0;\nbrev.b32 t, t;\nclz.b32 t, t;\nmin.u32 t, t, 31;\n" \
      "shfl.sync.idx.b32 need, a0, t, 31, 0xFFFFFFFF;\nsub.u32 need, need, t;\nadd.u32 m, need, lane;\n"      \
      "mov.u32 n, 0;\nmov.u32 r0, 0;\n" E(SR_OFF) E(SR_MAXR)                                                        \
      "setp.eq.and.u32 pf, n, 0, pa;\nsetp.lt.and.u32 pf, r0, awords, pf;\n"                \
      "vote.sync.all.pred pf, pf, 0xFFFFFFFF;\n@!pf bra.uni LSTGX;\nmov.u32 m, 0;\nand.b32 t, fl, 2;\nsetp.ne.u32 pf, t, 0;\nmov.u32 r5, 0;\n@pf bra.uni LRANGE;\n" \
      "LSTG1:\n" E(SR_STGV) "LSTG2:\n" "add.u32 gacc, gacc, cnt;\n" SR_FIN                                                     \
      /* stores of a block of several warps: publish the range from `need` on of space m and the stage, and wait    \
         until other warps have loaded in this round and lower ones with an overlapping store have stored */        \
      "LRANGE:\n"                                                                                                   \
      "and.b32 t, fl, 2304;\nsetp.eq.u32 pf, t, 256;\nselp.u32 qend, n32, 32 * " #V ", pf;\nadd.u32 qend, qend, need;\nsub.u32 qend, qend, 1;\n"                                                         \
      "LRANGE1:\nmad.lo.u32 t, " Q_W ", 16, " Q_GB ";\n"                                                              \
      "@pp st.shared.v4.u32 [t + " SR_STR(SR_GROUP_RANGE) "], {need, qend, m, m};\nadd.u32 keep, k4, 1;\n"                                       \
      "@pp st.release.cta.shared.u32 [myclk], keep;\nmad.lo.u32 t, lane, 16, " Q_GB ";\nmov.u32 n, 0;\n"              \
      "LRPOLL:\nld.acquire.cta.shared.u32 clk, [clks];\nld.shared.v4.u32 {r0, r1, r2, r3}, [t + " SR_STR(SR_GROUP_RANGE) "];\n"                  \
      "sub.u32 r4, clk, keep;\nsetp.ge.s32 pf, r4, 0;\nsetp.eq.u32 pa, r4, 0;\nsetp.lt.and.u32 pa, lane, " Q_W ", pa;\n" \
      "setp.eq.u32 pb, r2, m;\nsetp.eq.or.u32 pb, r2, 2, pb;\nand.pred pa, pa, pb;\n"                               \
      "setp.le.and.s32 pa, r0, qend, pa;\nsetp.le.and.s32 pa, need, r1, pa;\nnot.pred pa, pa;\nand.pred pf, pf, pa;\n" \
      "vote.sync.all.pred pf, pf, 0xFFFFFFFF;\n@pf bra.uni LRDONE;\n"                        \
      "add.u32 n, n, 1;\nld.shared.u32 u, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 28];\nsetp.ge.u32 pf, n, u;\n@pf bra.uni LTIMEOUT;\n"                                         \
      "setp.gt.u32 pf, n, 32;\n@pf nanosleep.u32 32;\nbra.uni LRPOLL;\n"                                            \
      "LRDONE:\nbar.warp.sync 0xFFFFFFFF;\nsetp.ne.u32 pa, r5, 0;\nsetp.ne.u32 pf, m, 0;\n"       \
      "@pa bra.uni LRDONE1;\n@pf bra.uni LSTS1;\nbra.uni LSTG1;\nLRDONE1:\n@!pf bra.uni LSTG3;\n"                   \
      /* stores consecutive within each slot (or one thread each): slot by slot, tids ascend with the slot */       \
      "LSTS3:\n" E(SR_STSO) "and.b32 t, fl, 131072;\nsetp.eq.u32 pf, t, 0;\n@pf bra.uni LSTS2;\n"                  \
      "ld.shared.u32 r0, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 64];\n" E(SR_WBS) "bra.uni LSTS2;\n"                                                                     \
      "LSTG3:\n" E(SR_STGO) "and.b32 t, fl, 262144;\nsetp.eq.u32 pf, t, 0;\n@pf bra.uni LSTG2;\n"                  \
      SR_GLOG(E, 1) "bra.uni LSTG2;\n"                                                                     \
      "LSTSX:\nsetp.lt.u32 pf, r0, sha;\nmov.u32 m, 1;\nvote.sync.all.pred pf, pf, 0xFFFFFFFF;\n@pf bra.uni LSTX;\n" \
      SR_REAL("131072", "r0", "12") "bra.uni LSTX;\n"                                  \
      "LSTGX:\nsetp.lt.u32 pf, r0, awords;\nmov.u32 m, 0;\nvote.sync.all.pred pf, pf, 0xFFFFFFFF;\n@pf bra.uni LSTX;\n" \
      SR_REAL("262144", "r0", "24")                                              \
      "LSTX:\n@!pf bra.uni LEND;\nsetp.ne.u32 pc, 0, 0;\n"                  \
      "mov.u32 need, 0x7FFFFFFF;\nmov.u32 qend, 0x80000000;\n" E(SR_OFF1)                                          \
      "vote.sync.any.pred pc, pc, 0xFFFFFFFF;\n@pc bra.uni LEND;\n"                                                \
      "redux.sync.min.s32 need, need, 0xFFFFFFFF;\nredux.sync.max.s32 qend, qend, 0xFFFFFFFF;\n"                   \
      "mov.u32 r5, 1;\nand.b32 t, fl, 2;\nsetp.ne.u32 pf, t, 0;\n@pf bra.uni LRANGE1;\nsetp.ne.u32 pf, m, 0;\n@pf bra.uni LSTS3;\n"       \
      "bra.uni LSTG3;\n"                                                                                           \
      /* 38 ATOMS */                                                                                                \
      "LMORE3:\nsetp.gt.u32 pf, u, 38;\n@pf bra.uni LMORE4;\nsetp.ge.s32 pf, fl, 0;\n@pf bra.uni LATOMS1;\n" SR_FLUSH(E, "C")              \
      "LATOMS1:\nprmt.b32 ro, x, 0, 0x4443;\n" SR_D_ROW "mad.lo.u32 ro, ro, " Q_STRIDE ", " Q_RS ";\n" LDB "mov.u32 m, 0;\n"    \
      E(SR_ADDR) E(SR_MAX)                                                                                          \
      "setp.lt.u32 pf, m, sha;\nvote.sync.all.pred pf, pf, 0xFFFFFFFF;\n@!pf bra.uni LATOMSU;\n"                    \
      "add.u32 need, k4, 2;\n@pp st.release.cta.shared.u32 [myclk], need;\n" SR_POLL("C")                           \
      "bar.warp.sync 0xFFFFFFFF;\n" E(SR_REDV) "LATOMS2:\n" SR_LOG(E, 2) TUP(E, 2) SR_FIN                         \
      "LATOMSU:\n" SR_REAL("131072", "m", "12") "@!pf bra.uni LEND;\nadd.u32 need, k4, 2;\n"                        \
      "@pp st.release.cta.shared.u32 [myclk], need;\n" SR_POLL("F") "bar.warp.sync 0xFFFFFFFF;\n" E(SR_REDV)         \
      "ld.shared.u32 r0, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 64];\n" E(SR_WBA) "bra.uni LATOMS2;\n"                                        \
      /* 39 BRA, 40 S2R, 41 BAR */                                                                                  \
      "LMORE4:\nsetp.eq.u32 pf, u, 39;\n@pf bra.uni LTAKE;\nsetp.eq.u32 pf, u, 40;\n@!pf bra.uni LMORE5;\n"         \
      SR_D_SREG "mad.lo.u32 t, y, 4, " Q_GB ";\nld.shared.u32 t, [t + " SR_STR(SR_GROUP_BV) " + 44];\nmov.u32 u, tid0;\nsetp.eq.u32 pa, y, 0;\n"    \
      E(SR_SREG) SR_ROW(STC, "LROWC", "LROWC1") SR_FIN                                                              \
      "LMORE5:\nand.b32 t, fl, 2056;\nsetp.eq.u32 pf, t, 8;\nsetp.eq.and.u32 pf, u, 41, pf;\n@!pf bra.uni LDIV;\n"     \
      "setp.ge.s32 pf, fl, 0;\n@pf bra.uni LBAR1;\n" SR_FLUSH(E, "D")       \
      "LBAR1:\nadd.u32 k4, k4, 4;\nand.b32 t, fl, 2;\nsetp.eq.u32 pf, t, 0;\n@pf bra.uni LBAR2;\n"                                                        \
      /* the park entry {waiting, exited, runnable, lowest pc} {highest pc, lowest runnable pc, round, flags} */    \
      "and.b32 r2, k4, 0x80000000;\nshr.u32 t, r2, 23;\nadd.u32 t, t, " Q_GB ";\nmad.lo.u32 u, " Q_W ", 32, t;\n"                               \
      "sub.u32 m, q, irs;\nshr.u32 m, m, 3;\nsub.u32 n, k4, r2;\nshr.u32 n, n, 2;\nmov.u32 r0, 0;\n"               \
      "mov.u32 need, n;\nmov.u32 r1, 0xFFFFFFFF;\nor.b32 r2, r2, 0x7FFFFFFF;\n"                                                      \
      "@pp st.shared.v4.u32 [u + " SR_STR(SR_GROUP_PARK) "], {n32, r0, r0, m};\n"                                   \
      "@pp st.shared.v4.u32 [u + " SR_STR(SR_GROUP_PARK) " + 16], {m, r1, n, r0};\n"                                \
      "@pp st.release.cta.shared.u32 [myclk], r2;\n"                                                               \
      "ld.shared.v4.u32 {r0, r1, t, r2}, [" Q_GB " + " SR_STR(SR_GROUP_CONST) " + 32];\nbar.sync 1, t;\n"         \
      "mov.u32 base, r2;\nmov.u32 bud, r0;\nand.b32 t, k4, 0x80000000;\nshr.u32 t, t, 23;\nadd.u32 t, t, " Q_GB ";\n"                                         \
      "and.b32 u, lane, 7;\nmad.lo.u32 u, u, 32, t;\n"                                                              \
      "ld.shared.v4.u32 {r0, r1, r2, r3}, [u + " SR_STR(SR_GROUP_PARK) "];\n"                                       \
      "ld.shared.v4.u32 {r4, r5, n, keep}, [u + " SR_STR(SR_GROUP_PARK) " + 16];\n"                                 \
      "or.b32 r1, r1, r2;\nor.b32 r1, r1, keep;\nsetp.ne.u32 pf, r0, 0;\nsetp.eq.and.u32 pf, r1, 0, pf;\n"          \
      "setp.eq.and.u32 pf, r3, m, pf;\nsetp.eq.and.u32 pf, r4, m, pf;\nsetp.ge.u32 pa, lane, base;\nor.pred pf, pf, pa;\n" \
      "selp.u32 n, 0, n, pa;\nredux.sync.max.u32 n, n, 0xFFFFFFFF;\nvote.sync.all.pred pf, pf, 0xFFFFFFFF;\n"       \
      "@!pf bra.uni LBARFULL;\nsub.u32 t, n, need;\nshl.b32 t, t, 2;\nadd.u32 kst, kst, t;\nand.b32 k4, k4, 0x80000000;\nxor.b32 k4, k4, 0x80000000;\nadd.u32 bud, bud, k4;\nmad.lo.u32 k4, n, 4, k4;\n" \
      "LBAR2:\nadd.u32 eh, eh, 64;\nsub.u32 k4, k4, 4;\n" SR_FIN                                                    \
      "LBARFULL:\nor.b32 fl, fl, 32768;\nbra.uni LDONE;\n"                                                                \
      /* 46 DIV, 48 REM by an immediate other than 0 and -1 */                                                      \
      "LDIV:\nsetp.eq.u32 pa, u, 46;\nsetp.eq.or.u32 pf, u, 48, pa;\n@!pf bra.uni LDIVR;\nadd.u32 t, y, 1;\n"        \
      "setp.gt.u32 pf, t, 1;\n@!pf bra.uni LEND;\n@!pa bra.uni LREM;\n" E(SR_DIVV) "LDIV1:\n"                      \
      SR_ROW(STC, "LROWD", "LROWD1") SR_FIN                                                                         \
      "LREM:\n" E(SR_REMV) "bra.uni LDIV1;\n"                                                                       \
      "LDIVR:\n" DIVR(E, LDB)                                                                                       \
      /* a chain's other factors and addends stand in the slots of its instructions, up to q */                     \
      "LCHAIN:\nsub.u32 t, t, 1;\nshl.b32 u, t, 3;\nsub.u32 u, q, u;\n"                                             \
      "setp.lt.u32 pf, t, 4;\n@pf bra.uni LCHAIN1;\n"                                                               \
      "LCHAIN4:\nld.shared.v2.u32 {m, n}, [u];\nld.shared.v2.u32 {r0, r1}, [u + 8];\n"                              \
      "ld.shared.v2.u32 {r2, r3}, [u + 16];\nld.shared.v2.u32 {r4, r5}, [u + 24];\n" E(SR_MAD) E(SR_MAD2) E(SR_MAD3) \
      E(SR_MAD4) "add.u32 u, u, 32;\nsub.u32 t, t, 4;\nsetp.ge.u32 pf, t, 4;\n@pf bra.uni LCHAIN4;\n"               \
      "LCHAIN1:\nsetp.eq.u32 pf, t, 0;\n@pf bra.uni LCHAINED;\n"                                                    \
      "ld.shared.v2.u32 {m, n}, [u];\n" E(SR_MAD) "add.u32 u, u, 8;\nsub.u32 t, t, 1;\nbra.uni LCHAIN1;\n"          \
      /* the other ALU groups */                                                                                    \
      "LGEN:\nadd.u32 q, q, 8;\n" SR_D_CODE("q") "ld.shared.v2.u32 {nx, ny}, [q];\n"                                                  \
      "prmt.b32 ro, x, 0, 0x4443;\n" SR_D_ROW "mad.lo.u32 ro, ro, " Q_STRIDE ", " Q_RS ";\nsetp.ge.u32 pf, u, 8;\n@pf bra.uni LREST;\n" \
      /* 3 MOV (operand b is zero), 4 ADD, 5 SUB, 6 MUL of registers */                                             \
      LDB "setp.eq.u32 pf, u, 5;\nselp.b32 m, 0xFFFFFFFF, 1, pf;\nsetp.eq.u32 pa, u, 6;\n" E(SR_REGOP)              \
      SR_TAIL(STC, "bra.uni LRUNEND;\n")                                                                            \
      "LREST:\n"                                                                                                    \
      E(SR_SPLAT) "and.b32 t, u, 1;\nsetp.ne.u32 pf, t, 0;\n@pf " LDB                                               \
      "setp.ge.u32 pf, u, 22;\n@pf bra.uni LCMP;\nsetp.ge.u32 pf, u, 14;\n@pf bra.uni LSHIFT;\n"                    \
      /* 8 AND, 10 OR, 12 XOR (+ 1: of registers) */                                                                \
      "setp.lt.u32 pa, u, 10;\nsetp.ge.u32 pb, u, 12;\nor.pred pc, pa, pb;\nnot.pred pc, pc;\n"                     \
      E(SR_LOGIC) SR_TAIL(STC, "bra.uni LRUNEND;\n")                                                                \
      "LSHIFT:\n" /* 14 SHL, 16 SHR, 18 MIN, 20 MAX */                                                              \
      "setp.lt.u32 pa, u, 16;\nsetp.ge.u32 pd, u, 20;\nsetp.ge.u32 pb, u, 18;\nnot.pred pc, pd;\n"                  \
      "and.pred pc, pc, pb;\nor.pred pb, pb, pa;\nnot.pred pb, pb;\n" E(SR_SHIFT)                                   \
      SR_TAIL(STC, "bra.uni LRUNEND;\n")                                                                            \
      "LCMP:\n" /* 22 SLT, 24 SLE, 26 SEQ, 28 SNE: (lt and pa) or (eq and pb), inverted under pc */                 \
      "setp.lt.u32 pa, u, 26;\nsetp.ge.u32 pb, u, 24;\nsetp.ge.u32 pc, u, 28;\n" E(SR_COMPARE)                      \
      SR_TAIL(STC, "bra.uni LRUNEND;\n")                                                                            \
      /* registers of some slots only */                                                                            \
      "LPART:\n@!ps bra.uni LNEXT;\n" E(SR_PUT)                                                                     \
      "LNEXT:\nmov.u32 x, nx;\nmov.u32 y, ny;\nmov.u32 keep, 64;\n@!pe bra.uni LALU;\nbra.uni LRUNEND;\n"           \
      "LROWA:\n@!ps bra.uni LROWA1;\n" E(SR_PUT) "bra.uni LROWA1;\n"                                                \
      "LROWB:\n@!ps bra.uni LROWB1;\n" E(SR_PUT) "bra.uni LROWB1;\n"                                                \
      "LROWD:\n@!ps bra.uni LROWD1;\n" E(SR_PUT) "bra.uni LROWD1;\n"                                                \
      "LROWC:\n@!ps bra.uni LROWC1;\n" E(SR_PUT) "bra.uni LROWC1;\n"                                                \
      SR_FLUSH_ANY(E, "A") SR_FLUSH_ANY(E, "B") SR_FLUSH_ANY(E, "C") SR_FLUSH_ANY(E, "D")                           \
      /* A branch forward that parts the threads: those that take it wait at its target, as the lowest-pc rule has   \
         it, while the others go on here, if every agent has some of these - or if a barrier or an exit stands at    \
         the target, where agents that take it as a whole wait in any case, and the budget has the round in which     \
         they come to wait there.  Not nested. */                                                                     \
      "LPARTS:\nsetp.eq.u32 pz, u, 34;\nsetp.ne.u32 pc, 0, 0;\n" E(SR_PARTS)                                        \
      SR_D_TARGET "mad.lo.u32 need, y, 8, irs;\nand.b32 t, fl, 512;\nsetp.ne.u32 pa, t, 0;\nsetp.gt.and.u32 pa, need, q, pa;\n"    \
      "setp.eq.and.u32 pa, qw, 0xFFFFFFF8, pa;\nld.shared.u32 t, [need];\nand.b32 t, t, 63;\nsetp.eq.u32 pb, t, 41;\n" \
      "setp.eq.or.u32 pb, t, 49, pb;\nadd.u32 t, k4, 8;\nsetp.le.and.u32 pb, t, bud, pb;\n"                         \
      "not.pred pd, pc;\nor.pred pb, pb, pd;\nand.pred pa, pa, pb;\n"                                              \
      "selp.u32 t, 14336, 10240, pc;\n@pa or.b32 fl, fl, t;\nbra.uni LEND;\n" /* (kSoloToNest, Nested, Agents) */  \
      "LNEST:\nadd.u32 k4, k4, 4;\nadd.u32 q, q, 8;\nand.b32 t, k4, 0x7FFFFFFF;\nsub.u32 u, t, kst;\nshr.u32 u, u, 2;\n" \
      "mad.lo.u32 ni, u, cnt, ni;\nmov.u32 kst, t;\nmov.u32 qw, need;\nmov.u32 x, nx;\nmov.u32 y, ny;\n"             \
      E(SR_NEST) "setp.ne.u32 pw, 0, 0;\nand.b32 fl, fl, 0xFFFFDFFF;\n"                                            \
      "bar.warp.sync 0xFFFFFFFF;\n@pp st.release.cta.shared.u32 [myclk], k4;\nbra.uni LMASK;\n"                     \
      /* the lowest waiting pc is reached: the waiting threads join again */                                        \
      "LSTOP:\nand.b32 t, fl, 2048;\nsetp.ne.u32 pa, t, 0;\nsetp.eq.and.u32 pa, q, qw, pa;\nsetp.lt.and.u32 pa, k4, bud, pa;\n" \
      "@pa or.b32 fl, fl, 16384;\nbra.uni LEND;\n"                                                                 \
      "LMERGE:\nand.b32 t, k4, 0x7FFFFFFF;\nsub.u32 u, t, kst;\nshr.u32 u, u, 2;\nmad.lo.u32 ni, u, cnt, ni;\n"      \
      "mov.u32 kst, t;\nmov.u32 qw, 0xFFFFFFF8;\nand.b32 fl, fl, 0xFFFFA7FF;\n" E(SR_JOIN) "mov.u32 wm, 0;\n"       \
      "and.b32 t, fl, 128;\nsetp.ne.u32 pw, t, 0;\nbra.uni LMASK;\n"                                               \
      "LTIMEOUT:\nor.b32 fl, fl, 65536;\n"                                                                         \
      "LEND:\nsetp.ge.s32 pf, fl, 0;\n@pf bra.uni LENDED;\n" SR_FLUSH(E, "B")                                      \
      "LENDED:\nand.b32 t, fl, 8192;\nsetp.ne.u32 pf, t, 0;\n@pf bra.uni LNEST;\n"                                 \
      "and.b32 t, fl, 16384;\nsetp.ne.u32 pf, t, 0;\n@pf bra.uni LMERGE;\n"                                        \
      "LDONE:\n" SR_D_DONE "and.b32 t, k4, 0x7FFFFFFF;\nsub.u32 u, t, kst;\nshr.u32 u, u, 2;\nmad.lo.u32 ni, u, cnt, ni;\n"       \
      "shl.b32 wm, wm, 4;\n" E(SR_OUT) "mov.u32 " Q_MASK ", wm;\nmov.u32 " Q_FL ", fl;\nmov.u32 " Q_QW ", qw;\n"     \
      "mov.u32 " Q_Q ", q;\nmov.u32 " Q_K4 ", k4;\nmov.u32 " Q_GACC ", gacc;\nmov.u32 " Q_SACC ", sacc;\n"           \
      "mov.u32 " Q_EH ", eh;\nmov.u32 " Q_NI ", ni;\n"                                                             \
      "}\n"                                                                                                         \
      : "+r"(q), "+r"(k4), "+r"(gacc), "+r"(sacc), "+r"(eh), "+r"(ni), "+r"(fl), "+r"(qw), "=r"(mask)               \
      : "r"(gb), "r"(w), "r"(rs), "r"(stride), "r"(am), "r"(fcap), "r"(bud)                                                 \
      : "memory")
// The numbers in the statement: places of what it reads, flags and masks, forms.
static_assert(offsetof(SoloConst, irs) == 0 && offsetof(SoloConst, rb) == 4 && offsetof(SoloConst, shs) == 8 &&
                  offsetof(SoloConst, sha) == 12 && offsetof(SoloConst, arena) == 16 && offsetof(SoloConst, arena_words) == 24 &&
                  offsetof(SoloConst, spin) == 28 && offsetof(SoloConst, budget4) == 32 && offsetof(SoloConst, nrows) == 36 &&
                  offsetof(SoloConst, nthr) == 40 && offsetof(SoloConst, nw) == 44 && offsetof(SoloConst, tup) == 48 &&
                  offsetof(SoloConst, tps4) == 52 && offsetof(SoloConst, region) == 56 && offsetof(SoloConst, wb) == 64 &&
                  offsetof(SoloConst, gcap) == 68 && offsetof(SoloConst, gblock) == 72 && offsetof(SoloConst, ncode) == 76 &&
                  offsetof(SoloConst, gregion) == 80,
              "constants in solo_loop");
static_assert(kGroupClk == 0 && 32 * kMaxWarps == 1 << (31 - 23) && kMaxWarps == 8, "clocks and park entries in solo_loop");
static_assert(kSoloPub == 1 && kSoloMany == 2 && kSoloLog == 4 && kSoloBar == 8 && kSoloFull == 16 && kSoloShared == 32 &&
                  kSoloGlobal == 64 && kSoloWhole == 128 && kSoloSolo == 512 && kSoloFused == 1024 && kSoloNested == 2048 &&
                  kSoloToNest == 8192 && kSoloToMerge == 16384 && kSoloAtBar == 32768 && kSoloTimeout == 65536 &&
                  kSoloUninit == 131072 && kSoloGlog == 262144 && kSoloBad == 0x80000 && kSoloPending == 0x80000000u &&
                  (kSoloLog | kSoloFull) == 20 && (kSoloSolo | kSoloPub) == 513 && (kSoloNested | kSoloBar) == 2056 &&
                  (kSoloNested | kSoloRegular) == 2304 && kSoloRegular == 256 && (kSoloToNest | kSoloNested) == 10240 &&
                  (kSoloToNest | kSoloNested | kSoloAgents) == 14336 && ~kSoloLog == 0xFFFFFFFBu && ~kSoloToNest == 0xFFFFDFFFu &&
                  ~(kSoloNested | kSoloAgents | kSoloToMerge) == 0xFFFFA7FFu && ~kSoloPending == 0x7FFFFFFFu,
              "flags in solo_loop");
static_assert(F_MULI == 2 && F_MOVR == 3 && F_SUBR == 5 && F_MULR == 6 && F_AND == 8 && F_OR == 10 && F_XOR == 12 && F_SHL == 14 &&
                  F_SHR == 16 && F_MIN == 18 && F_MAX == 20 && F_SLT == 22 && F_SLE == 24 && F_SEQ == 26 && F_SNE == 28 &&
                  F_LDS == 32 && F_STS == 33 && F_BRZ == 34 && F_BRNZ == 35 && F_LDG == 36 && F_STG == 37 && F_ATOMS == 38 &&
                  F_BRA == 39 && F_S2R == 40 && F_BAR == 41 && F_DIVI == 46 && F_REMI == 48 && F_EXIT == 49 && kFwdA == 64 &&
                  kDeadD == 128 && kNoDest == 31 && kRunMax == 255,
              "forms in solo_loop");

// Runs the set of the active slots `am` from instruction address q and clock k4 (4 * round with
// the interval's parity in bit 31) while it stays below the address qw and the clock below bud
// (with the parity too; when bud is other agents' round, a run of instructions that touch no memory
// goes on past it, uncut - its parts may be one chain - and unpublished there: at most 255 rounds);
// q, k4, eh (the epoch field of log records), fl (flags), qw and the per-lane counts of global and
// (fused) shared accesses and of executed instructions are updated.  gb: the block's shared memory;
// rs, stride: this lane's row 0 and the row stride; fcap: log records that fit.  Returns the slots
// active at the end, << 4 those that wait at qw.  Div: divisions by registers run here (with V = 4; in 64
// registers they would cost what does not divide 1%: the reduction of 2^24 values 2,490 us, with them
// 2,522).
template <int V, bool Fused, bool Div>
__device__ __forceinline__ uint32_t solo_loop(uint32_t& q, uint32_t& k4, uint32_t& gacc, uint32_t& sacc, uint32_t& eh,
                                              uint32_t& ni, uint32_t& fl, uint32_t& qw, uint32_t gb, uint32_t w,
                                              uint32_t rs, uint32_t stride, uint32_t am, uint32_t fcap, uint32_t bud) {
  uint32_t mask;
#define SR_SOLO_4(TUP, DIVR)                                                                                              \
  SR_SOLO_ASM(4, "c0, c1, c2, c3, b0, b1, b2, b3, a0, a1, a2, a3, l0, l1, l2, l3",                                  \
              "ld.shared.v4.u32 {c0, c1, c2, c3}, [ro];\n", "ld.shared.v4.u32 {b0, b1, b2, b3}, [ro];\n",           \
              "st.shared.v4.u32 [ro], {c0, c1, c2, c3};\n", "ld.shared.v4.u32 {a0, a1, a2, a3}, [ro];\n", SR_E4, TUP, DIVR)
#define SR_SOLO_2(TUP)                                                                                              \
  SR_SOLO_ASM(2, "c0, c1, b0, b1, a0, a1, l0, l1", "ld.shared.v2.u32 {c0, c1}, [ro];\n",                            \
              "ld.shared.v2.u32 {b0, b1}, [ro];\n", "st.shared.v2.u32 [ro], {c0, c1};\n",                           \
              "ld.shared.v2.u32 {a0, a1}, [ro];\n", SR_E2, TUP, SR_DIVR)
#define SR_SOLO_1(TUP)                                                                                              \
  SR_SOLO_ASM(1, "c0, b0, a0, l0", "ld.shared.u32 c0, [ro];\n", "ld.shared.u32 b0, [ro];\n",                        \
              "st.shared.u32 [ro], c0;\n", "ld.shared.u32 a0, [ro];\n", SR_E1, TUP, SR_DIVR)
  if constexpr (V == 4 && Fused && Div) SR_SOLO_4(SR_TUP, SR_DIVR);
  else if constexpr (V == 4 && Fused) SR_SOLO_4(SR_TUP, SR_NO_DIVR);
  else if constexpr (V == 4 && Div) SR_SOLO_4(SR_NO_TUP, SR_DIVR);
  else if constexpr (V == 4) SR_SOLO_4(SR_NO_TUP, SR_NO_DIVR);
  else if constexpr (V == 2 && Fused) SR_SOLO_2(SR_TUP);
  else if constexpr (V == 2) SR_SOLO_2(SR_NO_TUP);
  else if constexpr (Fused) SR_SOLO_1(SR_TUP);
  else SR_SOLO_1(SR_NO_TUP);
  return mask;
}
#undef SR_SOLO_1
#undef SR_SOLO_2
#undef SR_SOLO_4
#undef SR_SOLO_ASM

}  // namespace
}  // namespace sr
