// interp.cu - the SIMT interpreter: one real warp per 1, 2 or 4 simulated warps.
//
// What it computes (Hathhorn et al., SSV 2012): every thread of every block runs the
// kernel (Sec. 3 "Threads and memory"), blocks own a dynamic shared array (same
// section), __syncthreads() is a block-wide barrier (Sec. 3 "Barrier synchronization"),
// and every shared access is hooked (Sec. 3 "Modularity": the read/write check hook)
// - here the hook appends an 8-byte record to the block's access log for the race
// check of check.cu.  At each barrier the block's waiting threads are examined for
// divergence and deadlock (Sec. 3.1, last paragraph).
//
// GPU design.  A block's simulated warps are agents; a real warp runs V of them (block_vec), slot
// j of lane l being thread 32 (V w + j) + l, and nearly always executes one instruction for all
// of them at once: what bounds the interpreter is the latency and the issue slots of decoding
// and dispatch, and these are then paid once for V simulated warps.  A lane's V values of a
// register lie side by side (one 16-byte shared access for V = 4).  Registers, the simulated
// shared array and the program's code (staged by a TMA bulk copy) live in shared memory.
// Small blocks and small grids take a smaller V.  Instructions run in solo_loop (solo_loop.cuh); what it does not take -
// agents of a warp at different pcs, colliding or out-of-bounds addresses, barriers with
// something to report - runs in the general steps of run_block.
//
// The canonical schedule is round-lockstep across the block, but warps are NOT barrier-
// synchronised every round: each warp counts its own rounds (within a barrier interval
// an agent executes exactly one instruction per round while it has runnable threads) and
// publishes a logical clock 4*round + stage in shared memory.  Only memory
// instructions wait, and only for what the round semantics needs:
//   stage 0 (loads)   : every other warp has finished all earlier rounds;
//   stage 1 (stores)  : every other warp has done its loads of this round, and lower
//                       warps with an overlapping store in this round have stored
//                       (highest tid wins; within a warp via __match_any_sync);
//   stage 2 (atomics) : every other warp has done its stores of this round.
// ALU and branch instructions never wait, so warps drift freely between memory
// operations.  A clock carries the parity of its barrier interval in bit 31, and a warp whose
// threads all wait at a barrier or exited publishes the highest clock of its parity; then every
// warp reads all warps' park entries behind one CTA barrier, and if the release is plain all go
// on; otherwise warp 0 resolves it and a second CTA barrier follows.  Every wait is bounded
// (spin_limit) and reports SR_ST_INTERNAL instead of hanging.
//
// Measured (GB300, interpreter stage; before: one real warp per simulated warp, everything
// compiled C++): the reduction of 2^24 values 3,917 -> 1,521 us, 256 generated programs
// 19,912 -> 7,171 us, 96 of them with default shapes 5,893 -> 1,763 us, the 2048^2 stencil in 16
// launches 11,302 -> 5,563 us.
#include <algorithm>
#include <climits>

#include "solo_loop.cuh"
#include "sr_internal.h"

namespace sr {
namespace {

constexpr uint32_t FULL = 0xFFFFFFFFu;
enum : uint32_t { DEC_RELEASE = 1, DEC_DONE = 2, DEC_STOP = 3 };

struct BlockVars {
  uint32_t decision, any_race[2], n_misc;   // any_race: fused race check, words are marked (by interval parity)
  uint32_t cursor;             // log records reserved by the block (stops growing past the log)
  uint32_t flags, err_dirty, status;
  uint32_t bar_np, bar_nw;     // at a release: true predicates, released threads
  uint32_t race_out;           // fused race check: race entries written so far
  uint32_t gcursor;            // global-log records reserved by the block
  uint32_t sreg[4];            // S2R BID, BDIM, GDIM, WARPSIZE
};
static_assert(sizeof(BlockVars) <= 64, "block vars");
static_assert(offsetof(BlockVars, cursor) == 16 && offsetof(BlockVars, flags) == 20 && offsetof(BlockVars, gcursor) == 44 &&
                  offsetof(BlockVars, sreg) == 48 && BF_OVERFLOW == 1 && SR_SREG_TID == 0 && SR_SREG_BID == 1 &&
                  SR_SREG_BDIM == 2 && SR_SREG_GDIM == 3 && SR_SREG_WARPSIZE == 4 && K_R == 0 && K_W == 1 && K_A == 2,
              "block variables, registers and kinds in solo_loop");

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}
__device__ __forceinline__ uint32_t ld_acquire_gpu(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// ---- TMA bulk copy of the program code into shared memory (mbarrier completion)
__device__ __forceinline__ void mbar_init(unsigned long long* bar) {
  asm volatile("mbarrier.init.shared.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, unsigned long long* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, uint32_t phase, uint32_t limit) {
  for (uint32_t it = 0; it < limit; ++it) {
    uint32_t done;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Wait for the CTA's own code-staging copy.  Every thread polls; the CTA agrees on the
// outcome (__syncthreads_or), so that no thread takes a named barrier the others skip.  If the
// copy has not landed within kCopyWaitLimit polls it is waited for once more with the same
// bound; `drained` then says whether it has landed (the shared buffer and the mbarrier phase
// may be reused) or is still in flight (the CTA must leave both alone and exit).
__device__ __forceinline__ bool stage_wait(unsigned long long* bar, uint32_t phase, bool& drained) {
  const bool ok = !__syncthreads_or(!mbar_wait(bar, phase, kCopyWaitLimit));
  drained = ok || !__syncthreads_or(!mbar_wait(bar, phase, kCopyWaitLimit));
  return ok;
}

// A value that is the same in every lane, through a broadcast, which says so to the compiler.
__device__ __forceinline__ uint32_t same(uint32_t v) { return __shfl_sync(FULL, v, 0); }

// Shared-memory accesses by 32-bit shared-window address (cheaper address arithmetic than
// generic pointers in the interpreter's tight loops).
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts_u32(uint32_t a, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t lds_acquire(uint32_t a) {
  uint32_t v;
  asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
// The same under a predicate inside the statement.
__device__ __forceinline__ uint32_t lds_if(bool p, uint32_t a) {
  uint32_t v;
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %2, 0; mov.u32 %0, 0; @q ld.shared.u32 %0, [%1]; }"
               : "=&r"(v) : "r"(a), "r"((uint32_t)p) : "memory");
  return v;
}
__device__ __forceinline__ void sts_if(bool p, uint32_t a, uint32_t v) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q st.shared.u32 [%0], %1; }" ::"r"(a), "r"(v), "r"((uint32_t)p)
               : "memory");
}
__device__ __forceinline__ uint32_t atom_add_if(bool p, uint32_t a, uint32_t v, uint32_t otherwise) {
  uint32_t o;
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %3, 0; mov.u32 %0, %4; @q atom.shared.add.u32 %0, [%1], %2; }"
               : "=&r"(o) : "r"(a), "r"(v), "r"((uint32_t)p), "r"(otherwise) : "memory");
  return o;
}
__device__ __forceinline__ void st_release_if(bool p, uint32_t a, uint32_t v) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q st.release.cta.shared.u32 [%0], %1; }" ::"r"(a), "r"(v),
               "r"((uint32_t)p)
               : "memory");
}
__device__ __forceinline__ void sts_u128_if(bool p, uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t u) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %5, 0; @q st.shared.v4.u32 [%0], {%1, %2, %3, %4}; }" ::"r"(a), "r"(x),
               "r"(y), "r"(z), "r"(u), "r"((uint32_t)p)
               : "memory");
}
__device__ __forceinline__ uint32_t lds_u8(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint2 lds_u64(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
  return v;
}

// The simulated block's warps (named barrier 1: a CTA may hold warps that the block does not use).
__device__ __forceinline__ void block_sync(uint32_t nthr) {
  if (nthr == 32)
    __syncwarp();
  else
    asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
}

// Wait until every other warp of the block has published a clock >= need.  With
// `order` (store stage), also wait for lower warps whose store of this same round
// (clock == need) touches an overlapping range of the same memory space (ranges: {lowest,
// highest address, space, -} per warp).  clks: shared address of clock `lane`; pad: the lane
// stands for no other warp of the block.  Clocks and `need` carry the barrier interval's parity
// in bit 31, so that a warp still parked at the last barrier (other parity, all other bits set)
// reads as lower.
__device__ __forceinline__ bool wait_clocks(uint32_t clks, uint32_t ranges, bool pad, uint32_t w, uint32_t lane,
                                            uint32_t need, bool order, int32_t lo, int32_t hi, uint32_t sp,
                                            uint32_t limit) {
  for (uint32_t it = 0; it < limit; ++it) {
    const uint32_t c = lds_acquire(clks);
    bool ok = (int32_t)(c - need) >= 0;
    if (order) {
      int32_t l, h;
      uint32_t s;
      asm volatile("ld.shared.v2.u32 {%0, %1}, [%3];\nld.shared.u32 %2, [%3 + 8];"
                   : "=r"(l), "=r"(h), "=r"(s) : "r"(ranges + 16u * lane) : "memory");
      ok = ok && !(lane < w && c == need && (s == sp || s == 2u) && l <= hi && lo <= h);
    }
    if (__all_sync(FULL, ok || pad)) {
      __syncwarp();
      return true;
    }
    if (it >= 32) __nanosleep(32);
  }
  return false;
}

__device__ __forceinline__ void note_err(uint32_t* err, BlockVars* bv, uint32_t p, uint32_t w, uint32_t em,
                                         uint32_t lane) {
  if (lane == (uint32_t)(__ffs(em) - 1)) {
    atomicAdd(&err[2 * p], (uint32_t)__popc(em));
    atomicMin(&err[2 * p + 1], w * 32 + lane);
    bv->err_dirty = 1;
  }
}

// The 8-byte access-log record (layout in sr_internal.h) from its parts.
__device__ __forceinline__ unsigned long long rec_of(uint32_t epoch_hi, uint32_t low_bits, uint32_t addr) {
  return (unsigned long long)(epoch_hi | addr >> 8) << 32 | (low_bits | addr << 24);
}

// Append one 16-byte global-log record per lane with `me` to the block's global log (the
// same warp-aggregated reservation as log_wide).
__device__ __forceinline__ void log_global(BlockVars* bv, uint4* region, uint32_t cap, bool me, uint4 rec,
                                           uint32_t lane) {
  const uint32_t m = __ballot_sync(FULL, me);
  if (m == 0) return;
  const uint32_t leader = __ffs(m) - 1;
  uint32_t base = 0;
  if (lane == leader) {
    base = *reinterpret_cast<volatile uint32_t*>(&bv->gcursor);
    if (base < cap) base = atomicAdd(&bv->gcursor, (uint32_t)__popc(m));
  }
  base = __shfl_sync(FULL, base, leader);
  if (me) {
    const uint32_t pos = base + __popc(m & lanemask_lt());
    if (base < cap && pos < cap)
      region[pos] = rec;
    else
      atomicOr(&bv->flags, BF_OVERFLOW);
  }
}

// ---- fused race check (Sec. 3.1: each shared location keeps the accesses made to it since
// the last barrier).  The summary of a word: the two smallest distinct tids per access kind
// and the lowest and highest pc, enough to decide its races exactly.  Plane q of the
// summaries starts at tup + q * tps: planes 2k and 2k+1 hold the smallest and second
// smallest tid of kind k, planes 6 and 7 the pc range.  Every field is updated by one
// atomic min or max, so an access waits on at most one returned value.
//
// Lanes with `inb` add their access to word `addr`.  Inserting tid into (m1, m2): the min
// into m1 returns the old m1, and the larger of the two (unless equal or empty) is the
// candidate for m2; every value that leaves or misses m1 reaches m2, so m2 ends as the
// smallest tid different from m1.
__device__ __forceinline__ void tuple_add(uint32_t* tup, uint32_t tps, bool inb, uint32_t addr, uint32_t tid,
                                          uint32_t kind, uint32_t pc) {
  if (!inb) return;
  uint32_t* T = tup + addr;
  atomicMin(T + 6u * tps, pc);
  atomicMax(T + 7u * tps, pc);
  const uint32_t o = atomicMin(T + 2u * kind * tps, tid);
  if (o != tid && o != kTupleEmpty) atomicMin(T + (2u * kind + 1u) * tps, max(o, tid));
}

// Conflict classes and the smallest conflicting pair of a word from its summary (two threads
// conflict when distinct and write-write, write-read, write-atomic or atomic-read); false when
// the word has no race.
__device__ __forceinline__ bool tuple_race(const uint32_t* T, uint32_t tps, uint32_t& bout, uint32_t& cout) {
  const uint32_t R[2] = {T[0], T[tps]}, W[2] = {T[2u * tps], T[3u * tps]}, A[2] = {T[4u * tps], T[5u * tps]};
  uint32_t cls = 0, best = 0xFFFFFFFFu;
  auto pair = [&](uint32_t x, uint32_t y, uint32_t bit) {
    if (x == kTupleEmpty || y == kTupleEmpty || x == y) return;
    cls |= bit;
    best = min(best, min(x, y) << 16 | max(x, y));
  };
  pair(W[0], W[1], SR_CLS_WW);
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      pair(W[i], R[j], SR_CLS_WR);
      pair(W[i], A[j], SR_CLS_WA);
      pair(A[i], R[j], SR_CLS_AR);
    }
  if (!cls) return false;
  bout = best;
  cout = cls << 24 | (T[6u * tps] & 0xFFFu) << 12 | (T[7u * tps] & 0xFFFu);
  return true;
}

__device__ __forceinline__ void tuple_clear(uint32_t* T, uint32_t tps) {
#pragma unroll
  for (uint32_t q = 0; q < 7; ++q) T[q * tps] = kTupleEmpty;
  T[7u * tps] = 0;
}

// End of an interval, every warp of the block: words 32 j .. 32 j + 31 for its share of j.
// A racy word keeps its pair and class|pcs in planes 0 and 1 and is marked in the bitmap;
// every other touched word is cleared for the next interval.
__device__ __forceinline__ void tuples_mark(uint32_t* tup, uint32_t tps, uint32_t* rbm, uint32_t* any, uint32_t w,
                                            uint32_t nw, uint32_t lane) {
  const uint32_t nbw = tps / 32u;
  for (uint32_t j0 = w; j0 < nbw; j0 += 4u * nw) {
    uint32_t lo[4];                              // the lowest pcs: is the word touched?
#pragma unroll
    for (uint32_t i = 0; i < 4; ++i) {
      const uint32_t j = j0 + i * nw;
      lo[i] = j < nbw ? tup[6u * tps + 32u * j + lane] : kTupleEmpty;
    }
#pragma unroll 1
    for (uint32_t i = 0, j = j0; i < 4 && j < nbw; ++i, j += nw) {
      uint32_t* T = tup + 32u * j + lane;
      bool racy = false;
      if (lo[0] != kTupleEmpty) {
        uint32_t b, c;
        racy = tuple_race(T, tps, b, c);
        if (racy) {
          T[0] = b;
          T[tps] = c;
        } else {
          tuple_clear(T, tps);
        }
      }
      lo[0] = lo[1]; lo[1] = lo[2]; lo[2] = lo[3];
      const uint32_t m = __ballot_sync(FULL, racy);
      if (lane == 0) {
        rbm[j] = m;
        if (m) *any = 1u;
      }
    }
  }
}

// Warp 0: race entries of the interval's racy words in address order at the front of the
// block's region (16 bytes each, after the entries of earlier intervals), then the words are
// cleared.  A racy word had at least two accesses, so the entries fit wherever the region is
// sized by the accesses on a path; past `front_cap` record slots (a loop kernel's fixed
// region) entries are dropped and the block is flagged, as the access log would be.
__device__ void tuples_emit(uint32_t* tup, uint32_t tps, const uint32_t* rbm, BlockVars* bv,
                            unsigned long long* region, uint32_t front_cap, uint32_t epoch, uint32_t lane) {
  const uint32_t nbw = tps / 32u;
  const uint32_t cap = front_cap / 2u;           // entries that fit
  uint32_t ro = bv->race_out;
  bool over = false;
  uint4* out = reinterpret_cast<uint4*>(region);
  for (uint32_t base = 0; base < nbw; base += 32) {
    const uint32_t word = base + lane < nbw ? rbm[base + lane] : 0u;
    for (uint32_t nz = __ballot_sync(FULL, word != 0); nz; nz &= nz - 1u) {
      const uint32_t i = __ffs(nz) - 1, m = __shfl_sync(FULL, word, i);
      if ((m >> lane) & 1u) {
        const uint32_t a = (base + i) * 32u + lane, pos = ro + __popc(m & ((1u << lane) - 1u));
        uint32_t* T = tup + a;
        if (pos < cap)
          out[pos] = make_uint4(epoch, a, T[0], T[tps]);
        else
          over = true;
        tuple_clear(T, tps);
      }
      ro += __popc(m);
    }
  }
  ro = min(ro, cap);
  if (__any_sync(FULL, over) && lane == 0) bv->flags |= BF_OVERFLOW;
  __syncwarp();
  if (lane == 0) {
    bv->race_out = ro;
    bv->cursor = 2u * ro;                        // record slots the entries occupy
  }
  __syncwarp();
}

// Barrier/error records grow down from the end of the block's log region (16 B each).
__device__ void push_misc(BlockVars* bv, unsigned long long* region, uint32_t log_cap, uint32_t kind,
                          uint32_t epoch, uint32_t a, uint32_t b, uint32_t c) {
  const uint32_t i = bv->n_misc;
  const uint32_t used = bv->cursor < log_cap ? bv->cursor : log_cap;
  if (2ull * (i + 1) + used > log_cap) {
    bv->flags |= BF_OVERFLOW;
    return;
  }
  reinterpret_cast<uint4*>(region)[log_cap / 2 - 1 - i] = make_uint4(kind << 28 | epoch, a, b, c);
  bv->n_misc = i + 1;
}

// Error records of the interval, ordered by (kind, pc); run by one whole warp.
__device__ void flush_errors(BlockVars* bv, uint32_t* err, uint32_t* un, const uint2* ir, uint32_t ncode,
                             unsigned long long* region, uint32_t log_cap, uint32_t epoch, uint32_t lane) {
  const uint32_t last = un ? SR_REP_ERR_UNINIT_SHARED : SR_REP_ERR_DIV0;
  for (uint32_t kind = SR_REP_ERR_OOB_SHARED; kind <= last; ++kind) {
    for (uint32_t base = 0; base < ncode; base += 32) {
      const uint32_t pc = base + lane;
      uint32_t cnt = 0, mt = 0;
      bool hit = false;
      if (pc < ncode && kind == SR_REP_ERR_UNINIT_SHARED) {
        cnt = un[2 * pc];
        hit = cnt != 0;
        mt = un[2 * pc + 1];
      } else if (pc < ncode) {
        cnt = err[2 * pc];
        mt = err[2 * pc + 1];
        if (cnt && mt != kInf) {                 // (else the length of a run)
          const uint32_t f = pk_form(ir[pc].x);
          const uint32_t k2 = (f == F_LDS || f == F_STS || f == F_ATOMS) ? SR_REP_ERR_OOB_SHARED
                              : (f == F_LDG || f == F_STG)               ? SR_REP_ERR_OOB_GLOBAL
                                                                         : SR_REP_ERR_DIV0;
          hit = (k2 == kind);
        }
      }
      uint32_t hm = __ballot_sync(FULL, hit);
      while (hm) {
        const uint32_t j = __ffs(hm) - 1;
        hm &= hm - 1;
        const uint32_t jc = __shfl_sync(FULL, cnt, j), jm = __shfl_sync(FULL, mt, j);
        if (lane == 0) push_misc(bv, region, log_cap, kind, epoch, base + j, jm, jc);
        __syncwarp();
      }
    }
  }
  for (uint32_t pc = lane; pc <= ncode; pc += 32) {
    if (err[2 * pc + 1] != kInf) {
      err[2 * pc] = 0;
      err[2 * pc + 1] = kInf;
    }
    if (un) {
      un[2 * pc] = 0;
      un[2 * pc + 1] = kInf;
    }
  }
  __syncwarp();
  if (lane == 0) bv->err_dirty = 0;
}

// ---- one simulated thread per (lane, slot): warp w of a block runs the simulated warps
// V w .. V w + V - 1 ("agents"), slot j of its lane l being thread 32 (V w + j) + l.  A row of
// the register file holds a lane's V values side by side, so that one 4 V-byte access moves
// an operand of all of them.
template <int V>
__device__ __forceinline__ void lds_v(uint32_t a, uint32_t (&v)[V]) {
  if constexpr (V == 4)
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(a) : "memory");
  else if constexpr (V == 2)
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(a) : "memory");
  else
    v[0] = lds_u32(a);
}
template <int V>
__device__ __forceinline__ void sts_v(uint32_t a, const uint32_t (&v)[V]) {
  if constexpr (V == 4)
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
  else if constexpr (V == 2)
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(v[0]), "r"(v[1]) : "memory");
  else
    sts_u32(a, v[0]);
}
template <int V>
__device__ __forceinline__ void sts_v_if(bool p, uint32_t a, const uint32_t (&v)[V]) {
  if constexpr (V == 4)
    sts_u128_if(p, a, v[0], v[1], v[2], v[3]);
  else if constexpr (V == 2)
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %3, 0; @q st.shared.v2.u32 [%0], {%1, %2}; }" ::"r"(a), "r"(v[0]),
                 "r"(v[1]), "r"((uint32_t)p)
                 : "memory");
  else
    sts_if(p, a, v[0]);
}
// Row d of the active slots `am` (kNoDest: nothing): one store when every slot whose register
// still matters is active (`whole`, the same for the warp), else slot by slot.
template <int V>
__device__ __forceinline__ void put_row(uint32_t rs, uint32_t stride, uint32_t d, const uint32_t (&v)[V], uint32_t am,
                                        bool whole) {
  const uint32_t a = rs + d * stride;
  sts_v_if<V>(whole && d != kNoDest, a, v);
  if (!whole) {
#pragma unroll
    for (int j = 0; j < V; ++j) sts_if(((am >> j) & 1u) && d != kNoDest, a + 4u * j, v[j]);
  }
}

// A run of instructions for the general steps: as in solo_loop, from the one at shared
// address q with words (x, y) to the one before qend.  Returns the words at qend.
// rs + r * stride: this lane's row r; am: the slots to write when not all are (whole = 0).
#define SR_RPUT(i) "and.b32 t, %9, 1 << " #i ";\nsetp.ne.u32 pf, t, 0;\n@pf st.shared.u32 [ro + 4 * " #i "], c" #i ";\n"
// the result's store, and the next instruction or the end
#define SR_RTAIL(STC)                                                                                        \
  "setp.ge.u32 pe, q, %5;\n"                                                             \
  "and.b32 t, x, 128;\nsetp.eq.or.u32 ps, t, 0, pe;\n"                                                     \
  "prmt.b32 ro, x, 0, 0x4441;\nsetp.ne.and.u32 ps, ro, 31, ps;\nmad.lo.u32 ro, ro, %7, %6;\n"             \
  "@!pw bra.uni LPART;\n@ps " STC "mov.u32 x, nx;\nmov.u32 y, ny;\nmov.u32 keep, 64;\n"                    \
  "@!pe bra.uni LTOP;\nbra.uni LX;\n"
#define SR_RUN_ASM(REGS, LDC, LDB, STC, E)                                                                  \
  asm volatile(                                                                                             \
      "{\n"                                                                                                 \
      ".reg .pred pa, pb, pc, pd, pf, pe, ps, pw;\n.reg .b32 x, y, nx, ny, m, n, t, u, ro, keep, q;\n"      \
      ".reg .b32 " REGS ";\n"                                                                               \
      "mov.u32 x, %2;\nmov.u32 y, %3;\nmov.u32 q, %4;\nmov.u32 keep, 0;\nsetp.ne.u32 pw, %8, 0;\n"          \
      "LTOP:\n"                                                                                             \
      "and.b32 t, x, keep;\nsetp.eq.u32 pf, t, 0;\n"                                                        \
      "prmt.b32 ro, x, 0, 0x4442;\nmad.lo.u32 ro, ro, %7, %6;\n@pf " LDC                                    \
      "and.b32 u, x, 63;\nsetp.gt.u32 pf, u, 2;\n@pf bra.uni LGEN;\n"                                       \
      /* 0 MOV, 1 ADD, 2 MUL with an immediate: c * m + n */                                                \
      "prmt.b32 t, x, 0, 0x4443;\nmad.lo.u32 q, t, 8, q;\nld.shared.v2.u32 {nx, ny}, [q];\n"               \
      "setp.eq.u32 pf, u, 2;\nselp.u32 m, y, u, pf;\nselp.u32 n, 0, y, pf;\n" E(SR_MAD)                    \
      "sub.u32 t, t, 1;\nshl.b32 u, t, 3;\nsub.u32 u, q, u;\n"                                             \
      "LCHAIN:\nsetp.eq.u32 pf, t, 0;\n@pf bra.uni LCHAINED;\nld.shared.v2.u32 {m, n}, [u];\n" E(SR_MAD)  \
      "add.u32 u, u, 8;\nsub.u32 t, t, 1;\nbra.uni LCHAIN;\nLCHAINED:\n" SR_RTAIL(STC)                     \
      "LGEN:\nadd.u32 q, q, 8;\nld.shared.v2.u32 {nx, ny}, [q];\n"                                                                                             \
      "prmt.b32 ro, x, 0, 0x4443;\nmad.lo.u32 ro, ro, %7, %6;\nsetp.ge.u32 pf, u, 8;\n@pf bra.uni LREST;\n" \
      /* 3 MOV (operand b is zero), 4 ADD, 5 SUB, 6 MUL of registers */                                     \
      LDB "setp.eq.u32 pf, u, 5;\nselp.b32 m, 0xFFFFFFFF, 1, pf;\nsetp.eq.u32 pa, u, 6;\n" E(SR_REGOP)      \
      SR_RTAIL(STC)                                                                                          \
      "LREST:\n"                                                                                            \
      E(SR_SPLAT) "and.b32 t, u, 1;\nsetp.ne.u32 pf, t, 0;\n@pf " LDB                                       \
      "setp.ge.u32 pf, u, 22;\n@pf bra.uni LCMP;\nsetp.ge.u32 pf, u, 14;\n@pf bra.uni LSHIFT;\n"            \
      /* 8 AND, 10 OR, 12 XOR (+ 1: of registers) */                                                        \
      "setp.lt.u32 pa, u, 10;\nsetp.ge.u32 pb, u, 12;\nor.pred pc, pa, pb;\nnot.pred pc, pc;\n"             \
      E(SR_LOGIC) SR_RTAIL(STC)                                                                              \
      "LSHIFT:\n" /* 14 SHL, 16 SHR, 18 MIN, 20 MAX */                                                      \
      "setp.lt.u32 pa, u, 16;\nsetp.ge.u32 pd, u, 20;\nsetp.ge.u32 pb, u, 18;\nnot.pred pc, pd;\n"          \
      "and.pred pc, pc, pb;\nor.pred pb, pb, pa;\nnot.pred pb, pb;\n" E(SR_SHIFT) SR_RTAIL(STC)              \
      "LCMP:\n" /* 22 SLT, 24 SLE, 26 SEQ, 28 SNE: (lt and pa) or (eq and pb), inverted under pc */         \
      "setp.lt.u32 pa, u, 26;\nsetp.ge.u32 pb, u, 24;\nsetp.ge.u32 pc, u, 28;\n" E(SR_COMPARE) SR_RTAIL(STC) \
      "LPART:\n@!ps bra.uni LNEXT;\n" E(SR_RPUT)                                                             \
      "LNEXT:\nmov.u32 x, nx;\nmov.u32 y, ny;\nmov.u32 keep, 64;\n@!pe bra.uni LTOP;\n"                     \
      "LX:\nmov.u32 %0, x;\nmov.u32 %1, y;\n"                                                               \
      "}\n"                                                                                                 \
      : "=r"(out.x), "=r"(out.y)                                                                            \
      : "r"(x), "r"(y), "r"(q), "r"(qend), "r"(rs), "r"(stride), "r"(whole ? 1u : 0u), "r"(am)              \
      : "memory")
template <int V>
__device__ __forceinline__ uint2 alu_run(uint32_t x, uint32_t y, uint32_t q, uint32_t qend, uint32_t rs,
                                         uint32_t stride, bool whole, uint32_t am) {
  uint2 out;
  if constexpr (V == 4)
    SR_RUN_ASM("c0, c1, c2, c3, b0, b1, b2, b3", "ld.shared.v4.u32 {c0, c1, c2, c3}, [ro];\n",
               "ld.shared.v4.u32 {b0, b1, b2, b3}, [ro];\n", "st.shared.v4.u32 [ro], {c0, c1, c2, c3};\n", SR_E4);
  else if constexpr (V == 2)
    SR_RUN_ASM("c0, c1, b0, b1", "ld.shared.v2.u32 {c0, c1}, [ro];\n", "ld.shared.v2.u32 {b0, b1}, [ro];\n",
               "st.shared.v2.u32 [ro], {c0, c1};\n", SR_E2);
  else
    SR_RUN_ASM("c0, b0", "ld.shared.u32 c0, [ro];\n", "ld.shared.u32 b0, [ro];\n", "st.shared.u32 [ro], c0;\n", SR_E1);
  return out;
}
#undef SR_RUN_ASM

// Append one access record per slot of `im` to the block's log (one 32-bit shared atomic per
// warp and instruction; consecutive 8-byte slots, so coalesced stores).  `low` holds the low
// record bits of slot 0 without the address.  A warp that found the log full reserves nothing
// more, here or in solo_loop (entered without kSoloLog then), so the cursor cannot wrap.
template <int V>
__device__ __forceinline__ void log_wide(BlockVars* bv, unsigned long long* region, uint32_t front_cap, uint32_t im,
                                         const uint32_t (&ad)[V], uint32_t epoch_hi, uint32_t low, uint32_t lane,
                                         bool& full) {
  uint32_t total = 0, pos[V];
#pragma unroll
  for (int j = 0; j < V; ++j) {
    const uint32_t m = __ballot_sync(FULL, (im >> j) & 1u);
    pos[j] = total + __popc(m & lanemask_lt());
    total += __popc(m);
  }
  if (total == 0) return;
  const uint32_t base = same(atom_add_if(!full && lane == 0, smem_u32(&bv->cursor), total, 0xFFFFFFFFu));
  if (base >= front_cap || front_cap - base < total) {
    full = true;
    if (lane == 0) atomicOr(&bv->flags, BF_OVERFLOW);
  }
#pragma unroll
  for (int j = 0; j < V; ++j)
    if (((im >> j) & 1u) && base < front_cap && base + pos[j] < front_cap)
      region[base + pos[j]] = rec_of(epoch_hi, low + ((32u * j) << 14), ad[j]);
}

// Sum of a per-lane count over the warp (counts below 2^32, their sum may exceed it).
__device__ __forceinline__ unsigned long long warp_sum(uint32_t n) {
  return (unsigned long long)__reduce_add_sync(FULL, n & 0xFFFFu) +
         ((unsigned long long)__reduce_add_sync(FULL, n >> 16) << 16);
}

// Per-thread state word: pc (13 bits) | status << 16 | for a thread at a reducing barrier:
// destination row << 18 | kind (0 plain, 1 and, 2 or, 3 count) << 23 | predicate << 25.
__device__ __forceinline__ uint32_t ts_pc(uint32_t t) { return t & 0x1FFFu; }
__device__ __forceinline__ uint32_t ts_st(uint32_t t) { return (t >> 16) & 3u; }

// The start of a block, in the warps that run it: registers = params then zeros (the last row
// stays zero), shared memory and the block's records cleared.  Before the CTA waits for the
// launches it follows, and for its code; apart from run_block, whose registers it does not need.
template <int V, bool Fused>
__device__ __forceinline__ void start_block(const RunArgs& A, const LaunchDev* Ls, uint32_t block, const void* ir,
                                            unsigned char* gsm) {
  const uint32_t t = threadIdx.x, nw = Ls->nw, nthr = nw * 32u, sha = Ls->sha, ncode = Ls->ncode, nrows = Ls->nrows;
  const GroupLayout G = group_layout(nthr * V, sha, ncode, nrows, Ls->uninit, Ls->fused);
  const uint32_t rs = smem_u32(gsm + G.regs) + t * (4u * V), rstride = nthr * (4u * V);
  for (uint32_t r = 0; r < nrows; ++r) {
    uint32_t v[V];
#pragma unroll
    for (int j = 0; j < V; ++j) v[j] = r < Ls->nparams ? (uint32_t)Ls->params[r & 3u] : 0u;
    sts_v<V>(rs + r * rstride, v);
  }
  // error records: none (no tid), with the run lengths in place of the counts
  const uint8_t* runs = reinterpret_cast<const uint8_t*>(A.code + Ls->code_off) + ir_code_bytes(ncode);
  for (uint32_t i = t; i <= ncode; i += nthr) reinterpret_cast<uint2*>(gsm + G.err)[i] = make_uint2(__ldg(runs + i), kInf);
  auto fill4 = [&](uint32_t off, uint32_t words, uint32_t v) {
    for (uint32_t i = t; i < words / 4u; i += nthr) reinterpret_cast<uint4*>(gsm + off)[i] = make_uint4(v, v, v, v);
  };
  auto clear = [&](uint32_t off, uint32_t words) {
    for (uint32_t i = t; i < words; i += nthr) reinterpret_cast<uint32_t*>(gsm + off)[i] = 0;
  };
  fill4(G.sh, sha + 3u, 0);
  if (Ls->uninit) {
    for (uint32_t i = t; i <= ncode; i += nthr) reinterpret_cast<uint2*>(gsm + G.un)[i] = make_uint2(0u, kInf);
    clear(G.wb, (sha + 31u) / 32u);
  }
  const uint32_t tps = tuple_plane_words(sha);
  if (Fused && Ls->fused && A.check_races) {
    fill4(G.tup, 7u * tps, kTupleEmpty);
    fill4(G.tup + 28u * tps, tps, 0);
    clear(G.rbm, (sha + 31u) / 32u);
  }
  if ((t & 31u) == 0) reinterpret_cast<uint32_t*>(gsm + kGroupClk)[t >> 5] = 0;
  if (t == 0) {
    BlockVars* bv = reinterpret_cast<BlockVars*>(gsm + kGroupBv);
    bv->cursor = 0;
    bv->n_misc = 0; bv->flags = 0;
    bv->decision = 0; bv->err_dirty = 0; bv->status = 0;
    bv->race_out = 0;
    bv->any_race[0] = 0; bv->any_race[1] = 0;
    bv->gcursor = 0;
    bv->sreg[0] = block + Ls->block_off;
    bv->sreg[1] = Ls->bdim;
    bv->sreg[2] = Ls->gdim;
    bv->sreg[3] = 32u;
    SoloConst* sc = reinterpret_cast<SoloConst*>(gsm + kGroupConst);
    sc->irs = smem_u32(ir);
    sc->rb = smem_u32(gsm + G.err) - smem_u32(ir);
    sc->shs = smem_u32(gsm + G.sh);
    sc->sha = sha;
    sc->arena = reinterpret_cast<unsigned long long>(A.arena + Ls->arena_off);
    sc->arena_words = (uint32_t)Ls->arena_words;
    sc->spin = A.spin_limit;
    sc->budget4 = 4u * A.budget;
    if (kDebugBounds) {
      sc->nrows = nrows;
      sc->ncode = ncode;
    }
    sc->nthr = nthr;
    sc->nw = nw;
    sc->tup = smem_u32(gsm + G.tup);
    sc->tps4 = 4u * tps;
    sc->region = reinterpret_cast<unsigned long long>(A.log + Ls->log_base + (unsigned long long)block * Ls->log_cap);
    sc->wb = smem_u32(gsm + G.wb);
    sc->gcap = Ls->glog_cap;
    sc->gblock = Ls->block_base + block;
    sc->gregion = reinterpret_cast<unsigned long long>(A.glog + Ls->glog_base + (unsigned long long)block * Ls->glog_cap);
  }
}

// A launch is skipped when the launch before it in its stream, or the one it waits for,
// stopped or was skipped (Sec. 3, streams and events; Sec. 3.1, the interpreter halts).
__device__ __forceinline__ bool deps_dead(const RunArgs& A, const LaunchDev& L) {
  const volatile uint32_t* dead = A.launch_dead;
  return (L.dep_prev != kNoDep && dead[L.dep_prev]) || (L.dep_wait != kNoDep && dead[L.dep_wait]);
}

// Warp 0 of a CTA, batched mode: wait (bounded) until every block of the launches L follows
// (the previous launch of its stream, the one it waits for) has completed - they hold earlier
// places in the queue, so CTAs that never wait on L's blocks run them - and decide whether L is
// skipped (*skip set): a wait that gave up marks the program SR_ST_INTERNAL, and a launch that
// stopped or was skipped skips L (deps_dead).  A skipped launch is marked in launch_dead.
__device__ __forceinline__ void wait_deps(const RunArgs& A, const LaunchDev& L, uint32_t* skip) {
  bool give_up = false;
#pragma unroll 1
  for (uint32_t j = 0; j < 2 && !give_up; ++j) {
    const uint32_t dep = same(j ? L.dep_wait : L.dep_prev);
    if (dep == kNoDep) continue;
    const uint32_t need = same(A.launches[dep].grid);
    uint32_t s = 0;
    while (same(ld_acquire_gpu(&A.launch_done[dep])) < need) {
      if (++s >= A.spin_limit) {
        give_up = true;
        break;
      }
      __nanosleep(32);
    }
  }
  if (threadIdx.x == 0) {
    if (give_up) atomicOr(&A.prog_status[L.prog], (uint32_t)SR_ST_INTERNAL);
    if (give_up || deps_dead(A, L)) {
      atomicOr(&A.launch_dead[L.index], 1u);
      *skip = 1u;
    }
  }
  __syncwarp();
}

// (debug build) rounds that warps ran in solo_loop, for the test that it is what the build checks
#if defined(SR_DEBUG_BOUNDS)
__device__ unsigned long long g_loop_rounds;
__device__ __forceinline__ void note_loop(uint32_t rounds, uint32_t lane) {
  if (lane == 0) atomicAdd(&g_loop_rounds, (unsigned long long)rounds);
}
#else
__device__ __forceinline__ void note_loop(uint32_t, uint32_t) {}
#endif

// Run one simulated block on warps [0, Ls->nw) of the CTA, V simulated warps per warp.  The fused race check is compiled in only where Fused is set, and
// the logging of global accesses only where Global is set, so that the default kernels keep
// their register budget.
//
// Each agent (simulated warp) has its round count and next pc; the warp executes one
// instruction for a set of agents at the same pc and round.  Nearly always the set holds
// every agent that can run (`solo`): then only (p, k) are kept, in registers, and the decoding
// and dispatch of an instruction is paid once for V simulated warps.  Threads of an agent
// that wait at a higher pc for the lowest-pc rule to reach them do not end that (`wpc`: the
// lowest such pc).  Otherwise the agents' states sit in lanes 0..V-1 (ap next pc, ak round,
// aw lowest waiting pc) and the set with the lowest round runs, at one round first loads and
// everything that touches no memory, then stores, then atomics.
template <int V, bool Fused, bool Global, bool Div>
__device__ __forceinline__ void run_block(const RunArgs& A, const LaunchDev* Ls, uint32_t block,
                                          const uint2* __restrict__ ir, unsigned char* gsm) {
  const uint32_t w = same(threadIdx.x >> 5), nw = same(Ls->nw);
  constexpr uint32_t ALL = (1u << V) - 1u;
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t nthr = nw * 32;
  const uint32_t t = w * 32 + lane;              // thread of the group
  const uint32_t tid0 = w * 32 * V + lane;       // simulated thread of slot 0 (slot j: + 32 j)
  const uint32_t bdim = Ls->bdim, shw = same(Ls->shw), sha = same(Ls->sha), ncode = same(Ls->ncode), log_cap = same(Ls->log_cap);
  const uint32_t nrows = same(Ls->nrows);
  const bool uninit = same(Ls->uninit) != 0;
  const bool fused = Fused && same(Ls->fused) != 0 && A.check_races != 0;
  const GroupLayout G = group_layout(nthr * V, sha, ncode, nrows, Ls->uninit, Ls->fused);
  int32_t* sh = reinterpret_cast<int32_t*>(gsm + G.sh);
  uint32_t* clk = reinterpret_cast<uint32_t*>(gsm + kGroupClk);
  const uint32_t gb = same(smem_u32(gsm)), clks = gb + kGroupClk + 4u * lane, myclk = gb + kGroupClk + 4u * w;
  const uint32_t ranges = gb + kGroupRange;
  const bool pad = lane >= nw || lane == w;      // (of wait_clocks)
  uint32_t* err = reinterpret_cast<uint32_t*>(gsm + G.err);
  uint32_t* un = reinterpret_cast<uint32_t*>(gsm + G.un);      // with `uninit` only
  uint32_t* wb = reinterpret_cast<uint32_t*>(gsm + G.wb);      // with `uninit` only
  uint32_t* tup = reinterpret_cast<uint32_t*>(gsm + G.tup);    // with `fused` only
  const uint32_t tps = tuple_plane_words(sha);
  uint32_t* rbm = reinterpret_cast<uint32_t*>(gsm + G.rbm);
  BlockVars* bv = reinterpret_cast<BlockVars*>(gsm + kGroupBv);
  int32_t* arena = A.arena + Ls->arena_off;
  const uint32_t arena_words = same((uint32_t)Ls->arena_words);
  unsigned long long* region = A.log + Ls->log_base + (unsigned long long)block * log_cap;
  const bool logging = A.check_races != 0;
  // global log of this block (with Global, for launches whose glog_cap is set)
  const uint32_t gcap = Global ? Ls->glog_cap : 0u;
  const uint32_t gblock = Ls->block_base + block;
  uint4* gregion = Global ? A.glog + Ls->glog_base + (unsigned long long)block * gcap : nullptr;
  const uint32_t budget = A.budget, spin = A.spin_limit;
  // 32-bit shared-window addresses: row r of this lane is at rs + r * rstride
  const uint32_t rs = smem_u32(gsm + G.regs) + t * (4u * V), rstride = nthr * (4u * V);
  const uint32_t shs = smem_u32(sh), irs = smem_u32(ir);
  const bool pub = lane == 0 && nw > 1;          // this thread publishes the warp's clock

  uint32_t ts[V], xm = 0;                        // state words; xm: slots without a thread, or exited
  uint32_t p = same(Ls->entry), k = 0, wpc = kInf;     // the running set: pc, round, lowest waiting pc
#pragma unroll
  for (int j = 0; j < V; ++j) {
    const bool none = tid0 + 32u * j >= bdim;
    ts[j] = p | (none ? ST_NONE : ST_RUN) << 16;
    xm |= (none ? 1u : 0u) << j;
  }
  uint32_t am = ALL & ~xm;                       // its active slots of this lane
  // every slot whose registers still matter is active; ns: slots 0 .. ns - 1 are active in every
  // lane and no others (0: the active threads form no such shape)
  bool whole;
  uint32_t ns;
  auto set_shape = [&]() {
    whole = __all_sync(FULL, (am | xm) == ALL);
    const uint32_t m = same(am);
    ns = __all_sync(FULL, am == m) && (m & (m + 1u)) == 0 ? __popc(m) : 0u;
  };
  set_shape();
  uint32_t nexit = 0;                            // exited threads of the warp
  bool errs = false;                             // the warp noted errors in this interval
  uint32_t sub = ALL;                            // its agents
  bool solo = true;                              // it holds every agent that can run
  uint32_t ak = 0, ap = kInf, aw = kInf;         // lanes 0..V-1: the agents, while not solo
  uint32_t epoch = 0, front_cap = log_cap;
  uint32_t par = 0;                              // the barrier interval's parity, in bit 31
  uint32_t n_instr = 0, n_gacc = 0;              // per lane: executed instructions, global accesses
  uint32_t n_sacc = 0;                           // per lane, fused race check: shared accesses
  bool lfull = false;
  // a log record is built from 32-bit halves: low = addr << 24 | tid << 14 | kind << 12 | pc,
  // high = epoch << 6 | addr >> 8
  const uint32_t lane_rec = tid0 << 14;
  uint32_t epoch_hi = 0;                         // epoch << 6
  enum : uint32_t { GO, PICK, RESCHED };
  uint32_t how = GO;
  uint32_t kn = 0;                               // not solo: the lowest round of the other agents, if memory may be
                                                 // accessed in the rounds below it (else 0)
  const uint32_t solo_flags = (nw > 1 ? kSoloMany : 0u) | (logging && !fused ? kSoloLog : 0u) | (fused ? kSoloFused : 0u);
  const uint32_t solo_mem = (uninit ? kSoloUninit : kSoloShared) | (Global && gcap ? kSoloGlog : kSoloGlobal);

  // (debug build) every row of the run of `len` instructions at p is in the register file
  auto rows_ok = [&](uint32_t p, uint32_t len) {
    bool ok = true;
    if (kDebugBounds)
      for (uint32_t q = p, x; q < p + len; q += pk_form(x) <= F_MULI ? pk_b(x) : 1u) {
        x = ir[q].x;
        ok = ok && dbg_ok(q < ncode && pk_a(x) < nrows && (pk_imm(pk_form(x)) || pk_b(x) < nrows) &&
                              (pk_d(x) < nrows || pk_d(x) == kNoDest),
                          &A.prog_status[Ls->prog], SR_ST_BOUNDS);
      }
    return ok;
  };

  for (;;) {  // barrier intervals
    bool at_bar = false;                         // the warp's threads wait at barrier p, their states not written
    uint32_t stop = 0;                           // 1: out of rounds, 2: a wait gave up
    for (;;) {  // steps of the running set
      bool multi_st = false;                     // stores of other pcs share this round
      bool moved = false;                        // solo_loop ran some instructions
      if (how != GO) {
        if (how == RESCHED) {                    // the agents' next and waiting pcs from the threads'
#pragma unroll
          for (int j = 0; j < V; ++j) {
            const uint32_t c = ts_st(ts[j]) == ST_RUN ? ts_pc(ts[j]) : kInf;
            const uint32_t m = __reduce_min_sync(FULL, c);
            const uint32_t m2 = __reduce_min_sync(FULL, c != m ? c : kInf);
            if (lane == (uint32_t)j) {
              ap = m;
              aw = m2;
            }
          }
        }
        const uint32_t can = __ballot_sync(FULL, ap != kInf);
        if (!can) break;
        k = __reduce_min_sync(FULL, ap != kInf ? ak : kInf);
        if (k >= budget) {
          stop = 1;
          break;
        }
        const bool cand = ap != kInf && ak == k;
        p = __shfl_sync(FULL, ap, __ffs(__ballot_sync(FULL, cand)) - 1);
        sub = __ballot_sync(FULL, cand && ap == p);
        solo = sub == can;
        kn = 0;
        if (!solo) {
          // among the agents at this round: what touches no memory, then loads, one pc at a time;
          // then stores (agent by agent when they are at several pcs); then atomics
          uint32_t cls = 4;
          if (cand) {
            const uint32_t o = pk_form(ir[ap].x);
            cls = (o == F_LDS || o == F_LDG) ? 1u : (o == F_STS || o == F_STG) ? 2u : o == F_ATOMS ? 3u : 0u;
          }
          const uint32_t first = __reduce_min_sync(FULL, cls);
          const uint32_t of = __ballot_sync(FULL, cls == first);
          p = __shfl_sync(FULL, ap, __ffs(of) - 1);
          sub = __ballot_sync(FULL, cls == first && ap == p);
          if (first == 2 && (sub != of || clk[w] == 4u * k + 1u + par)) {
            multi_st = true;                     // (also for the last of them)
            sub &= 0u - sub;
          }
          // the only set at this round, about to access memory: it may, in the rounds up to the
          // others' lowest (as long as nothing of this round is published; away from the budget,
          // which runs of the set may pass otherwise)
          const uint32_t o = same(pk_form(ir[p].x));
          kn = __reduce_min_sync(FULL, ap != kInf && !((sub >> lane) & 1u) ? ak : kInf);
          if (kn == k || multi_st || same(clk[w]) > 4u * k + par || kn + 256u > budget || o < F_LDS || o > F_ATOMS ||
              o == F_BRZ || o == F_BRNZ)
            kn = 0;
        }
        wpc = __reduce_min_sync(FULL, (sub >> lane) & 1u ? aw : kInf);
        am = 0;
#pragma unroll
        for (int j = 0; j < V; ++j)
          if (((sub >> j) & 1u) && ts_st(ts[j]) == ST_RUN && ts_pc(ts[j]) == p) am |= 1u << j;
        set_shape();
        __syncwarp();
        st_release_if(pub && 4u * k + par > clk[w], myclk, 4u * k + par);
        how = GO;
      } else if (k >= budget) {                  // (solo)
#pragma unroll
        for (int j = 0; j < V; ++j)
          if ((am >> j) & 1u) ts[j] = p;
        ak = k;
        stop = 1;
        break;
      }
      {
        // Most instructions run in solo_loop; what it does not take is left at (p, k).  While other
        // agents are at later rounds, it runs up to their lowest; with some at the same round, it runs
        // ahead over what touches no memory.
        const uint32_t k_in = k;
        uint32_t q = same(irs + p * 8u), k4 = same(4u * k + par), eh = same(epoch_hi);
        uint32_t qw = same(wpc == kInf ? 0xFFFFFFF8u : irs + wpc * 8u);
        uint32_t fl = solo_flags | (whole ? kSoloWhole : 0u) | (ns ? kSoloRegular : 0u);
        if (lfull) fl = (fl & ~kSoloLog) | kSoloFull;
        if (solo) fl |= kSoloSolo;
        if (solo || kn) fl |= kSoloPub | solo_mem;
        if (solo && whole && nexit == 0 && !errs && !fused && wpc == kInf) fl |= kSoloBar;
        fl = same(fl);
        const uint32_t mask = solo_loop<V, Fused, Div>(q, k4, n_gacc, n_sacc, eh, n_instr, fl, qw, gb, w, rs, rstride, am,
                                                  same(front_cap), same(4u * (solo || !kn ? budget : kn) + par));
        fl = same(fl);
        lfull = (fl & kSoloFull) != 0;
        p = (same(q) - irs) >> 3;
        k4 = same(k4);
        par = k4 & 0x80000000u;
        k = (k4 - par) >> 2;
        epoch_hi = same(eh);
        epoch = epoch_hi >> 6;
        moved = k != k_in;
        if (kDebugBounds) {
          note_loop(k - k_in, lane);
          if (fl & kSoloBad) {                   // stop the block the way a wait that gave up does
            if (lane == 0) atomicOr(&A.prog_status[Ls->prog], (uint32_t)SR_ST_BOUNDS);
            if (!(fl & kSoloAtBar)) {
              stop = 2;
              break;
            }
          }
        }
        if (fl & kSoloNested) {
          // some threads wait at a higher pc (at a barrier or exit: agents without a running thread
          // have executed it)
          wpc = (same(qw) - irs) >> 3;
          am = mask & ALL;
          const bool exits = pk_form(lds_u64(irs + wpc * 8u).x) == F_EXIT;
          uint32_t gone = 0;
#pragma unroll
          for (int j = 0; j < V; ++j) {
            const bool at = (fl & kSoloAgents) && !__any_sync(FULL, (am >> j) & 1u);
            if ((mask >> (4 + j)) & 1u) {
              ts[j] = !at ? wpc : exits ? wpc | ST_EXIT << 16 : (wpc + 1u) | ST_WAIT << 16;
              n_instr += at;
              gone |= (at && exits ? 1u : 0u) << j;
            }
          }
          if (exits) {
            xm |= gone;
            nexit += __reduce_add_sync(FULL, __popc(gone));
          }
          set_shape();
        }
        if (fl & kSoloAtBar) {
          at_bar = true;
          break;
        }
        if (fl & kSoloTimeout) {
          stop = 2;
          break;
        }
        if (solo && k >= budget) continue;
      }
      const uint2 in = lds_u64(irs + p * 8u);
      const uint32_t f = pk_form(in.x);
      // (what touches no memory may run ahead of other agents' earlier rounds)
      if (p < wpc && (solo || !moved || (k < budget && (f > F_ATOMS || f == F_BRZ || f == F_BRNZ)))) {
      const uint32_t run = f < F_LDS ? lds_u8(smem_u32(err) + 8u * p) : 0u;
      if (run) {
        // A run of instructions that touch no memory and do not branch executes in a tight loop,
        // one instruction per round; its last round is published at once (other warps wait on
        // a clock only for memory effects).
        const uint32_t len = min(min(run, budget - k), wpc - p);
        if (!rows_ok(p, len)) {                  // stop the block the way a wait that gave up does
          stop = 2;
          break;
        }
        st_release_if(solo && pub, myclk, 4u * (k + len) + par);
        alu_run<V>(in.x, in.y, irs + p * 8u, irs + (p + len) * 8u, rs, rstride, whole, am);
        n_instr += len * __popc(am);
        p += len;
        k += len;
      } else {
        const uint32_t d = pk_d(in.x), ra = rs + pk_a(in.x) * rstride, rb = rs + pk_b(in.x) * rstride;
        const uint32_t imm = in.y;
        if (!dbg_ok(p <= ncode && pk_a(in.x) < nrows && pk_b(in.x) < nrows && (d < nrows || d == kNoDest),
                    &A.prog_status[Ls->prog], SR_ST_BOUNDS)) {
          stop = 2;                              // (debug build) stop the block like a failed wait
          break;
        }
        n_instr += __popc(am);
        if (f <= F_STS || (f >= F_LDG && f <= F_ATOMS)) {
          const bool shared = f != F_LDG && f != F_STG;
          const uint32_t bound = shared ? sha : arena_words;
          uint32_t ad[V], im = 0;                // addresses; im: active slots whose address is in bounds
          bool past = false;                     // a shared address in bounds that shared_reach ruled out
          lds_v<V>(ra, ad);
#pragma unroll
          for (int j = 0; j < V; ++j) {
            ad[j] += imm;
            im |= (ad[j] < bound ? 1u : 0u) << j;
            past = past || (((am >> j) & 1u) && shared && ad[j] >= sha && ad[j] < shw);
          }
          im &= am;
          if (__any_sync(FULL, past)) {          // (never: stop the block rather than leave it out)
            stop = 2;
            break;
          }
          uint32_t kind = K_R;
          if (f == F_LDS || f == F_LDG) {
            if (nw > 1 && !wait_clocks(clks, ranges, pad, w, lane, 4u * k + par, false, 0, 0, 0, spin)) {
              stop = 2;
              break;
            }
            uint32_t v[V];
#pragma unroll
            for (int j = 0; j < V; ++j) {
              const bool me = (im >> j) & 1u;
              v[j] = lds_if(me && shared, shs + ad[j] * 4u);
              if (me && !shared) v[j] = (uint32_t)arena[ad[j]];
            }
            put_row<V>(rs, rstride, d, v, am, whole);
            if (shared && uninit) {              // words no store or atomic of an earlier round wrote
#pragma unroll
              for (int j = 0; j < V; ++j) {
                const uint32_t um = __ballot_sync(
                    FULL, ((im >> j) & 1u) && !((wb[ad[j] >> 5] >> (ad[j] & 31u)) & 1u));
                if (um) {
                  errs = true;
                  note_err(un, bv, p, w * V + j, um, lane);
                }
              }
            }
          } else if (f == F_ATOMS) {
            kind = K_A;
            uint32_t v[V];
            lds_v<V>(rb, v);
            if (nw > 1) {
              st_release_if(pub, myclk, 4u * k + 2u + par);
              if (!wait_clocks(clks, ranges, pad, w, lane, 4u * k + 2u + par, false, 0, 0, 0, spin)) {
                stop = 2;
                break;
              }
            }
#pragma unroll
            for (int j = 0; j < V; ++j)
              if ((im >> j) & 1u) atomicAdd(&sh[ad[j]], (int32_t)v[j]);
          } else {
            kind = K_W;
            uint32_t v[V];
            lds_v<V>(rb, v);
            if (nw > 1) {
              int32_t lo = INT_MAX, hi = INT_MIN;
#pragma unroll
              for (int j = 0; j < V; ++j)
                if ((im >> j) & 1u) {
                  lo = min(lo, (int32_t)ad[j]);
                  hi = max(hi, (int32_t)ad[j]);
                }
              lo = __reduce_min_sync(FULL, lo);
              hi = __reduce_max_sync(FULL, hi);
              // stores of several pcs in this round: any address of either space, from the first on
              sts_u128_if(pub, ranges + 16u * w, (uint32_t)(multi_st ? INT_MIN : lo), (uint32_t)(multi_st ? INT_MAX : hi),
                          multi_st ? 2u : shared ? 1u : 0u, 0u);
              st_release_if(pub, myclk, 4u * k + 1u + par);
              if (!wait_clocks(clks, ranges, pad, w, lane, 4u * k + 1u + par, true, lo, hi, shared ? 1u : 0u, spin)) {
                stop = 2;
                break;
              }
            }
            // Several threads on one word: the highest tid's store is the one kept.  Consecutive
            // addresses (address - tid equal over the storing threads) cannot collide; any other
            // pattern stores slot by slot (tids ascend with the slot), in each slot the highest
            // lane of a word.
            const uint32_t m0 = __ballot_sync(FULL, im & 1u);
            const uint32_t ref = __shfl_sync(FULL, ad[0] - lane, m0 ? __ffs(m0) - 1 : 0);
            bool consec = m0 != 0 || !(im & 1u);
#pragma unroll
            for (int j = 0; j < V; ++j) consec = consec && (!((im >> j) & 1u) || ad[j] - lane - 32u * j == ref);
            if (m0 != 0 && __all_sync(FULL, consec)) {
#pragma unroll
              for (int j = 0; j < V; ++j)
              {
                const bool me = (im >> j) & 1u;
                sts_if(me && shared, shs + ad[j] * 4u, v[j]);
                if (me && !shared) arena[ad[j]] = (int32_t)v[j];
              }
            } else {
#pragma unroll
              for (int j = 0; j < V; ++j) {
                const bool me = (im >> j) & 1u;
                const uint32_t m = __ballot_sync(FULL, me);
                if (m) {
                  const uint32_t off = __shfl_sync(FULL, ad[j] - lane, __ffs(m) - 1);
                  bool last = me;
                  if (!__all_sync(FULL, !me || ad[j] - lane == off)) {
                    const uint32_t grp = __match_any_sync(FULL, me ? ad[j] : (0x80000000u | lane));
                    last = me && lane == 31u - __clz(grp);
                  }
                  sts_if(last && shared, shs + ad[j] * 4u, v[j]);
                  if (last && !shared) arena[ad[j]] = (int32_t)v[j];
                  __syncwarp();
                }
              }
            }
          }
          if (shared && uninit && kind != K_R) {
#pragma unroll
            for (int j = 0; j < V; ++j)
              if ((im >> j) & 1u) atomicOr(&wb[ad[j] >> 5], 1u << (ad[j] & 31u));
          }
          if (__any_sync(FULL, im != am)) {
            errs = true;
#pragma unroll
            for (int j = 0; j < V; ++j) {
              const uint32_t em = __ballot_sync(FULL, ((am & ~im) >> j) & 1u);
              if (em) note_err(err, bv, p, w * V + j, em, lane);
            }
          }
          if (shared) {
            if (fused) {
#pragma unroll
              for (int j = 0; j < V; ++j) tuple_add(tup, tps, (im >> j) & 1u, ad[j], tid0 + 32u * j, kind, p);
              n_sacc += __popc(im);
            } else if (logging) {
              log_wide<V>(bv, region, front_cap, im, ad, epoch_hi, lane_rec | kind << 12 | p, lane, lfull);
            }
          } else {
            n_gacc += __popc(am);
            if (Global && gcap) {
#pragma unroll
              for (int j = 0; j < V; ++j)
                log_global(bv, gregion, gcap, (im >> j) & 1u,
                           make_uint4(ad[j], epoch, (tid0 + 32u * j) << 16 | kind << 12 | p, gblock), lane);
            }
          }
          ++p;
          ++k;
          // every lane's access is ordered before the clock (warp barrier, then a release)
          __syncwarp();
        } else if (f >= F_DIVR && f <= F_REMI) {
          uint32_t a[V], b[V], zm = 0;
          lds_v<V>(ra, a);
          if (f == F_DIVI || f == F_REMI) {
#pragma unroll
            for (int j = 0; j < V; ++j) b[j] = imm;
          } else {
            lds_v<V>(rb, b);
          }
#pragma unroll
          for (int j = 0; j < V; ++j) {
            const int32_t x = (int32_t)a[j], y = (int32_t)b[j];
            const int32_t s = (y == 0 || y == -1) ? 1 : y;   // (INT_MIN / -1 would trap)
            const int32_t qt = x / s;
            if (y == 0) {
              zm |= 1u << j;
              a[j] = 0u;
            } else if (f <= F_DIVI) {
              a[j] = y == -1 ? 0u - (uint32_t)x : (uint32_t)qt;   // -INT_MIN wraps to INT_MIN
            } else {
              a[j] = y == -1 ? 0u : (uint32_t)(x - qt * s);
            }
          }
          put_row<V>(rs, rstride, d, a, am, whole);
          zm &= am;
          if (__any_sync(FULL, zm != 0)) {
            errs = true;
#pragma unroll
            for (int j = 0; j < V; ++j) {
              const uint32_t em = __ballot_sync(FULL, (zm >> j) & 1u);
              if (em) note_err(err, bv, p, w * V + j, em, lane);
            }
          }
          ++p;
          ++k;
        } else if (f == F_S2R) {
          const uint32_t u = imm == SR_SREG_BID    ? block + Ls->block_off
                             : imm == SR_SREG_BDIM ? bdim
                             : imm == SR_SREG_GDIM ? Ls->gdim
                                                   : 32u;
          uint32_t v[V];
#pragma unroll
          for (int j = 0; j < V; ++j) v[j] = imm == SR_SREG_TID ? tid0 + 32u * j : u;
          put_row<V>(rs, rstride, d, v, am, whole);
          ++p;
          ++k;
        } else if (f == F_BRA) {
          p = imm;
          ++k;
        } else if (f == F_BRZ || f == F_BRNZ) {
          uint32_t a[V], tm = 0;                 // tm: active slots that take the branch
          lds_v<V>(ra, a);
#pragma unroll
          for (int j = 0; j < V; ++j) tm |= ((a[j] == 0) == (f == F_BRZ) ? 1u : 0u) << j;
          tm &= am;
          ++k;
          if (!__any_sync(FULL, tm != 0)) {
            ++p;
          } else if (!__any_sync(FULL, tm != am)) {
            p = imm;
          } else {                               // both ways: the threads' pcs part
#pragma unroll
            for (int j = 0; j < V; ++j)
              if ((am >> j) & 1u) ts[j] = (tm >> j) & 1u ? imm : p + 1u;
            if ((sub >> lane) & 1u) ak = k;
            how = RESCHED;
            continue;
          }
        } else {
          // barriers: the thread waits; a reducing form hands in its predicate and keeps the row
          // its result goes to.  EXIT, and the EXIT sentinel after the last instruction.
          const bool bar = f != F_EXIT;
          uint32_t a[V];
#pragma unroll
          for (int j = 0; j < V; ++j) a[j] = 0;
          uint32_t word = p | ST_EXIT << 16;
          if (bar) {
            word = (p + 1u) | ST_WAIT << 16;
            if (f != F_BAR) {
              lds_v<V>(ra, a);
              word |= d << 18 | (f - F_BAR) << 23;
            }
          } else {
            xm |= am;
            nexit += __reduce_add_sync(FULL, __popc(am));
          }
#pragma unroll
          for (int j = 0; j < V; ++j)
            if ((am >> j) & 1u) ts[j] = word | (a[j] != 0 ? 1u << 25 : 0u);
          ++k;
          if ((sub >> lane) & 1u) ak = k;
          if (solo && wpc == kInf) break;        // no thread of the warp can run
          how = RESCHED;
          continue;
        }
      }
      // (p, k): the set's next instruction
      if (solo && p < wpc) {
        st_release_if(pub, myclk, 4u * k + par);
        continue;
      }
      }
#pragma unroll
      for (int j = 0; j < V; ++j)
        if ((am >> j) & 1u) ts[j] = p;
      if ((sub >> lane) & 1u) {
        ak = k;
        ap = p;
      }
      how = p < wpc ? PICK : RESCHED;
    }

    // ---- no runnable thread in this warp (or it stopped): publish its state and park
    // (`uni`: every waiting thread at one barrier pc and none runnable, the usual case: they
    // all resume together after that barrier)
    bool uni = at_bar;
    uint32_t upc = p;
    const uint32_t parks = gb + kGroupPark + (par ? 32u * kMaxWarps : 0u);   // the interval's park entries
    if (!at_bar) {                               // (else solo_loop wrote it and passed the CTA barrier)
      uint32_t n = 0, np = 0, mn = kInf, mx = 0, rp = kInf;   // counts: wait | exit << 10 | run << 20
#pragma unroll
      for (int j = 0; j < V; ++j) {
        const uint32_t st = ts_st(ts[j]), c = ts_pc(ts[j]);
        if (st == ST_WAIT) {
          n += 1u;
          np += ts[j] >> 25 | ((ts[j] >> 23) & 3u ? 1u << 16 : 0u);   // predicates; reducing barriers << 16
          mn = min(mn, c - 1u);
          mx = max(mx, c - 1u);
        } else if (st == ST_EXIT) {
          n += 1u << 10;
        } else if (st == ST_RUN) {
          n += 1u << 20;
          rp = min(rp, c);
        }
      }
      n = __reduce_add_sync(FULL, n);
      np = __reduce_add_sync(FULL, np);
      mn = __reduce_min_sync(FULL, mn);
      mx = __reduce_max_sync(FULL, mx);
      rp = __reduce_min_sync(FULL, rp);
      const uint32_t kx = __reduce_max_sync(FULL, lane < (uint32_t)V ? ak : 0u);
      uni = (n >> 20) == 0 && (n & 0x3FFu) != 0 && mn == mx;
      upc = mn;
      sts_u128_if(lane == 0, parks + 32u * w, n & 0x3FFu, (n >> 10) & 0x3FFu, n >> 20, mn);
      sts_u128_if(lane == 0, parks + 32u * w + 16u, mx, rp, kx, stop | (errs ? 4u : 0u) | np << 8);
      st_release_if(pub, myclk, par | 0x7FFFFFFFu);
      block_sync(nthr);
    }
    if (fused) {                                 // the interval's touched words, all warps
      tuples_mark(tup, tps, rbm, &bv->any_race[par >> 31], w, nw, lane);
      block_sync(nthr);
    }

    // ---- barrier resolution.  Every thread of the block waits at one plain barrier and there is
    // nothing to report: each warp sees that in the park entries and goes on by itself (the other
    // interval's entries are written next, so none is overwritten while a warp still reads it).
    // Otherwise warp 0 resolves the barrier and a second CTA barrier follows.
    const bool v = lane < nw;
    uint4 pa, pb;                                // warp `lane`'s entry
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(pa.x), "=r"(pa.y), "=r"(pa.z), "=r"(pa.w) : "r"(parks + 32u * (lane & 7u)) : "memory");
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(pb.x), "=r"(pb.y), "=r"(pb.z), "=r"(pb.w) : "r"(parks + 32u * (lane & 7u) + 16u) : "memory");
    const uint32_t kmax = __reduce_max_sync(FULL, v ? pb.z : 0u);
    const uint32_t pc0 = same(pa.w);
    const bool racy = fused && same(bv->any_race[par >> 31]);   // (cleared behind the second barrier)
    if (!racy && __all_sync(FULL, !v || (pa.x && !(pa.y | pa.z | pb.w) && pa.w == pc0 && pb.x == pc0))) {
      epoch += 1u;
    } else if (!racy && __all_sync(FULL, !v || !(pa.x | pa.z | pb.w))) {
      break;                                     // every thread exited, nothing to report
    } else {
      if (w == 0) {
        const uint32_t nW = __reduce_add_sync(FULL, v ? pa.x : 0u);
        const uint32_t nX = __reduce_add_sync(FULL, v ? pa.y : 0u);
        const uint32_t nR = __reduce_add_sync(FULL, v ? pa.z : 0u);
        const uint32_t pmn = __reduce_min_sync(FULL, v ? pa.w : kInf);
        const uint32_t pmx = __reduce_max_sync(FULL, v ? pb.x : 0u);
        const uint32_t rpc = __reduce_min_sync(FULL, v ? pb.y : kInf);
        const uint32_t fl = __reduce_or_sync(FULL, v ? pb.w & 0xFFu : 0u);
        const uint32_t nP = __reduce_add_sync(FULL, v ? (pb.w >> 8) & 0xFFFFu : 0u);
        if (racy) tuples_emit(tup, tps, rbm, bv, region, log_cap - 2u * bv->n_misc, epoch, lane);
        uint32_t dec = DEC_RELEASE, kind = 0, a = 0, b = 0, c = 0, stbits = 0;
        if (fl & 2u) {
          dec = DEC_STOP;
          if (lane == 0) bv->flags |= BF_INTERNAL;
        } else if (fl & 1u) {          // out of rounds
          dec = DEC_STOP; kind = SR_REP_STEP_LIMIT; a = budget; b = nR; c = rpc; stbits = SR_ST_STEP_LIMIT;
        } else if (nW == 0) {          // every thread exited
          dec = DEC_DONE;
        } else if (nX > 0) {           // some wait at a barrier that exited threads never reach
          dec = DEC_STOP; kind = SR_REP_DEADLOCK; a = pmn; b = pmx; c = nW << 16 | nX; stbits = SR_ST_DEADLOCK;
        } else if (pmn != pmx) {       // all wait: release, flag differing barrier pcs
          kind = SR_REP_DIVERGENCE; a = pmn; b = pmx; c = nW << 16;
        }
        if (lane == 0 && kind) push_misc(bv, region, log_cap, kind, epoch, a, b, c);
        __syncwarp();
        if (bv->err_dirty) flush_errors(bv, err, uninit ? un : nullptr, ir, ncode, region, log_cap, epoch, lane);
        if (lane == 0) {
          bv->decision = dec;
          bv->status |= stbits;
          bv->bar_np = nP;
          bv->bar_nw = nW;
        }
      }
      block_sync(nthr);
      if (same(bv->decision) != DEC_RELEASE) break;
      if (t == 0) bv->any_race[par >> 31] = 0;   // (marked again behind the next CTA barrier at the earliest)
      front_cap = log_cap - 2u * same(bv->n_misc);
      epoch += 1u;
    }
    k = ak = kmax;
    par ^= 0x80000000u;
    errs = false;
    epoch_hi = epoch << 6;
    st_release_if(pub, myclk, 4u * k + par);
    if (at_bar) {
      ++p;                                       // (the set stays as it is)
    } else {
      am = 0;
#pragma unroll
      for (int j = 0; j < V; ++j)
        if (ts_st(ts[j]) == ST_WAIT) {
          // a reducing barrier's result, over every released thread's predicate
          const uint32_t kind = (ts[j] >> 23) & 3u, row = (ts[j] >> 18) & 31u;
          if (kind && row != kNoDest) {
            const uint32_t np = bv->bar_np;
            sts_u32(rs + row * rstride + 4u * j,
                    kind == 1 ? (np == bv->bar_nw ? 1u : 0u) : kind == 2 ? (np ? 1u : 0u) : np);
          }
          ts[j] = ts_pc(ts[j]);                  // runs on after its barrier
          am |= 1u << j;
        }
      set_shape();
      how = RESCHED;
      if (uni) {                                 // every released thread resumes after its barrier
        p = upc + 1u;
        wpc = kInf;
        sub = ALL;
        solo = true;
        how = GO;
      }
    }
  }

  // ---- block finished
  const unsigned long long wi = warp_sum(n_instr), wg = warp_sum(n_gacc);
  const unsigned long long ws = Fused ? warp_sum(n_sacc) : 0ull;
  if (lane == 0) {
    atomicAdd(&A.counters->thread_instrs, wi);
    if (wg) atomicAdd(&A.counters->global_accesses, wg);
    if (ws) atomicAdd(&A.counters->shared_accesses, ws);
  }
  if (t == 0) {
    const uint32_t front = log_cap - 2u * bv->n_misc;
    BlockRes r;
    r.n_log = fused ? 0u : (bv->cursor < front ? bv->cursor : front);   // fused: no records to check
    r.n_race = fused ? bv->race_out : 0u;
    r.n_misc = bv->n_misc;
    r.flags = bv->flags;
    A.blocks[Ls->block_base + block] = r;
    if (Global && gcap) {
      const uint32_t ng = bv->gcursor < gcap ? bv->gcursor : gcap;
      A.glog_n[gblock] = ng;
      if (ng) atomicAdd(&A.counters->global_records, (unsigned long long)ng);
    }
    if (r.n_log) atomicAdd(&A.counters->shared_accesses, (unsigned long long)r.n_log);
    const uint32_t bits = bv->status | ((bv->flags & BF_OVERFLOW) ? (uint32_t)SR_ST_LOG_OVERFLOW : 0u) |
                          ((bv->flags & BF_INTERNAL) ? (uint32_t)SR_ST_INTERNAL : 0u);
    if (bits) atomicOr(&A.prog_status[Ls->prog], bits);
    if (bits & (SR_ST_DEADLOCK | SR_ST_STEP_LIMIT | SR_ST_INTERNAL)) atomicOr(&A.launch_dead[Ls->index], 1u);
  }
}

// Warp 0 of a CTA: its launch's descriptor into shared memory.
__device__ __forceinline__ void copy_launch(LaunchDev* dst, const LaunchDev* src) {
  static_assert(sizeof(LaunchDev) % 4 == 0, "copied by words");
  for (uint32_t i = threadIdx.x; i < sizeof(LaunchDev) / 4; i += 32)
    reinterpret_cast<uint32_t*>(dst)[i] = __ldg(reinterpret_cast<const uint32_t*>(src) + i);
  __syncwarp();
}

// The CTA's block once its launch is known and its code is under way: clear, wait for the code,
// run (unless warp 0 has found, before it comes here, that the launch is skipped).
template <int V, bool Fused, bool Global, bool Div>
__device__ __forceinline__ void run_staged(const RunArgs& A, const LaunchDev* Ls, uint32_t block, unsigned char* smem,
                                           unsigned long long* mbar, const uint32_t* skip) {
  // every thread must take the same branch before the block's named barriers
  const bool mine = __all_sync(FULL, (threadIdx.x >> 5) < Ls->nw);
  if (mine) start_block<V, Fused>(A, Ls, block, smem, smem + Ls->ir_bytes);
  bool drained;
  if (!__any_sync(FULL, stage_wait(mbar, 0, drained))) {           // (its barrier also ends the clearing)
    if (threadIdx.x == 0) atomicOr(&A.prog_status[Ls->prog], (uint32_t)SR_ST_INTERNAL);
  } else if (mine && !same(*skip)) {
    run_block<V, Fused, Global, Div>(A, Ls, block, reinterpret_cast<const uint2*>(smem), smem + Ls->ir_bytes);
  }
}

// One CTA per simulated block; one kernel launch per (program, launch), in an order that
// respects every stream and wait.  A block takes block_warps(bdim, V) warps: at most 8 with
// V = 2 and 4, two with V = 1 (block_vec).  MINB: CTAs of that many warps the registers allow.
template <int V, int MINB, bool Fused, bool Global>
__global__ void __launch_bounds__(V == 1 ? 64 : 256, MINB) k_interp_plain(RunArgs A, uint32_t li) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ LaunchDev Ls;
  __shared__ __align__(8) unsigned long long mbar;
  __shared__ uint32_t s_skip;
  if (threadIdx.x < 32) {
    copy_launch(&Ls, A.launches + li);
    if (threadIdx.x == 0) {
      // (the launches before this one have completed: they ran earlier on this CUDA stream)
      s_skip = deps_dead(A, Ls);
      if (s_skip) atomicOr(&A.launch_dead[Ls.index], 1u);
      if (!s_skip) {
        mbar_init(&mbar);
        bulk_load(smem, A.code + Ls.code_off, Ls.ir_bytes, &mbar);
      }
    }
  }
  __syncthreads();
  if (same(s_skip)) return;
  run_staged<V, Fused, Global, MINB != 4>(A, &Ls, blockIdx.x, smem, &mbar, &s_skip);
}

// Batched mode: the blocks of many launches in one grid, one simulated block per CTA.  The host
// puts launches together that take the same kernel form and warps and about the same shared
// memory (a bucket), so that the CTAs an SM holds follow from what these blocks need; the
// buckets of a wave run side by side on streams of their own.  A block's place in the bucket's
// queue is its ticket: where launches follow others, the CTAs take tickets from a counter, in
// the order of launch level, launch and block, so that the launches a block's launch follows
// hold smaller tickets, taken by CTAs that are already running, and the CTA waits for them
// (bounded); else it is the CTA's index.  No loop surrounds the block and its warps are chosen
// by a warp vote: a persistent loop around it cost several hundred bytes of spills.
template <int V, int MINB, bool Fused, bool Global>
__global__ void __launch_bounds__(V == 1 ? 64 : 256, MINB) k_interp_blocks(RunArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ LaunchDev Ls;
  __shared__ __align__(8) unsigned long long mbar;
  __shared__ uint32_t s_skip, s_bad, s_block, s_li;
  if (threadIdx.x < 32) {
    const uint32_t lane = threadIdx.x;
    uint32_t t = blockIdx.x;
    if (A.bq_head) {                                // one ticket per CTA: t < the grid size
      if (lane == 0) t = atomicAdd(A.bq_head, 1u);
      t = __shfl_sync(FULL, t, 0);
    }
    // the queue entry holding ticket t: the last one whose first ticket is <= t; the lanes probe
    // 32 places of [lo, hi) at a time
    uint32_t lo = 0, hi = A.bq_n;
    while (hi - lo > 1) {
      const uint32_t step = (hi - lo + 31u) / 32u, at = lo + lane * step;
      const uint32_t m = __ballot_sync(FULL, at < hi && __ldg(A.bq_first + at) <= t);   // (lane 0 always)
      const uint32_t last = 31u - __clz(m);
      lo += last * step;
      hi = min(hi, lo + step);
    }
    const uint32_t li = A.bq_launch[lo];
    copy_launch(&Ls, A.launches + li);
    if (lane == 0) {
      s_li = li;
      s_block = t - A.bq_first[lo];
      const bool bad = s_block >= Ls.grid;          // (a corrupt queue: never from load_programs)
      if (bad) {
        atomicOr(&A.prog_status[Ls.prog], (uint32_t)SR_ST_INTERNAL);
      } else {
        mbar_init(&mbar);
        bulk_load(smem, A.code + Ls.code_off, Ls.ir_bytes, &mbar);
      }
      s_bad = bad ? 1u : 0u;
      s_skip = 0;
    }
    __syncwarp();
    // the other warps clear their part of the block's memory while this one waits
    asm volatile("bar.arrive 2, %0;" ::"r"(blockDim.x) : "memory");
    if (A.bq_head && !same(s_bad)) wait_deps(A, Ls, &s_skip);
  } else {
    asm volatile("bar.sync 2, %0;" ::"r"(blockDim.x) : "memory");
  }
  if (!same(s_bad)) run_staged<V, Fused, Global, MINB != 4>(A, &Ls, s_block, smem, &mbar, &s_skip);
  if (!A.bq_head) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&A.launch_done[s_li], 1u);
  }
}

}  // namespace

#if defined(SR_DEBUG_BOUNDS)
// Of the debug build alone: rounds that warps have run in the interpreter's inner loop.
extern "C" int sr_debug_loop_rounds(unsigned long long* out) {
  return cudaMemcpyFromSymbol(out, g_loop_rounds, sizeof *out) == cudaSuccess ? SR_OK : SR_E_CUDA;
}
#endif

uint32_t interp_plain_smem(const LaunchDev& L) {
  return L.ir_bytes + group_layout(L.nw * 32u * L.vec, L.sha, L.ncode, L.nrows, L.uninit, L.fused).total;
}

// dynamic shared memory may use what the kernel's static shared memory leaves of the opt-in limit
template <typename K>
static cudaError_t allow_dynamic_smem(K kernel, uint32_t smem_optin) {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(smem_optin - (uint32_t)fa.sharedSizeBytes));
}

// The kernels: simulated warps per warp x register budget x fused race check x global log.
typedef void (*PlainKernel)(RunArgs, uint32_t);
typedef void (*BlocksKernel)(RunArgs);
template <int V, int MINB>
static PlainKernel plain_of(bool fused, bool global) {
  if (global) return k_interp_plain<V, MINB, false, true>;
  return fused ? k_interp_plain<V, MINB, true, false> : k_interp_plain<V, MINB, false, false>;
}
static PlainKernel plain_kernel(uint32_t vec, uint32_t variant, bool fused, bool global) {
  if (vec == 1) return plain_of<1, 12>(fused, global);
  if (vec == 2) return plain_of<2, 3>(fused, global);
  return variant == 2 ? plain_of<4, 4>(fused, global) : plain_of<4, 3>(fused, global);
}
template <int V, int MINB>
static BlocksKernel blocks_of(bool fused, bool global) {
  if (global) return k_interp_blocks<V, MINB, false, true>;
  return fused ? k_interp_blocks<V, MINB, true, false> : k_interp_blocks<V, MINB, false, false>;
}
static BlocksKernel blocks_kernel(uint32_t vec, uint32_t variant, bool fused, bool global) {
  if (vec == 1) return blocks_of<1, 12>(fused, global);
  if (vec == 2) return blocks_of<2, 3>(fused, global);
  return variant == 2 ? blocks_of<4, 4>(fused, global) : blocks_of<4, 3>(fused, global);
}

cudaError_t init_interp_attributes(uint32_t smem_optin) {
  cudaError_t e = cudaSuccess;
  for (uint32_t vec = 1; vec <= 4 && e == cudaSuccess; vec *= 2)
    for (uint32_t variant = 1; variant <= (vec == 4 ? 2u : 1u) && e == cudaSuccess; ++variant)
      for (uint32_t f = 0; f < 3 && e == cudaSuccess; ++f) {
        e = allow_dynamic_smem(plain_kernel(vec, variant, f == 1, f == 2), smem_optin);
        if (e == cudaSuccess) e = allow_dynamic_smem(blocks_kernel(vec, variant, f == 1, f == 2), smem_optin);
      }
  return e;
}

// variant: 1 = the larger register budget, 2 = more CTAs per SM (and more spills), 0 = 2 where its CTAs
// fit and warps wait much: at four barriers or more.  The reduction of 2^24 values (11 barriers)
// 1,592 us with 1 and 1,500 with 2, 1501 blocks of 333 threads 81 and 58; 64 generated programs (most
// with one to three) 1,738 and 1,906, the 2048^2 stencil (one) 5,532 and 6,770.  Intervals of one store
// and 2 to 12 ALU instructions in full grids, time with 1 over time with 2: blocks of 256 threads 0.92 to
// 0.94 at one barrier, 0.97 to 1.07 at three, 1.02 to 1.10 at four, 1.09 to 1.12 at eight; of 1024 threads
// 0.90 to 0.92, 0.94 to 1.00, 0.96 to 1.02, 1.02 to 1.05.  A kernel with a loop counts as without
// barriers: with 24 turns of two barriers each it would be 1.06 to 1.10 times as fast with 2.
cudaError_t launch_interp_plain(const RunArgs& a, uint32_t li, const LaunchDev& L, uint32_t variant,
                                uint32_t smem_per_sm, cudaStream_t s) {
  const uint32_t threads = L.nw * 32u;
  const uint32_t smem = interp_plain_smem(L);
  const bool global = L.glog_cap != 0;
  const bool fused = L.fused != 0 && !global;
  if (variant == 0)
    variant = L.barriers >= 4 && std::min(32u / L.nw, smem_per_sm / (smem + kBlocksStaticSmem)) > 24u / L.nw ? 2 : 1;
  plain_kernel(L.vec, variant, fused, global)<<<L.grid, threads, smem, s>>>(a, li);
  return cudaGetLastError();
}

cudaError_t launch_interp_blocks(const RunArgs& a, uint32_t vec, uint32_t variant, uint32_t warps, uint32_t nblocks,
                                 uint32_t smem, bool fused, bool global, cudaStream_t s) {
  blocks_kernel(vec, variant, fused, global)<<<nblocks, warps * 32u, smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace sr
