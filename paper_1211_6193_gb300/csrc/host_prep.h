// host_prep.h - host-side preparation of simulated programs shared by the entry points of
// libsimtcheck: validation, register renaming, instruction packing and the static bound
// of a kernel's per-block access log.  Internal; not part of the C ABI.
#pragma once
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <vector>
#include <cuda_runtime.h>
#include <stdint.h>

#include "simtcheck.h"
#include "sr_internal.h"

namespace sr {
namespace host {

// barriers: __syncthreads and its reducing forms _and / _or / _count
inline bool is_barrier(uint32_t b) { return b == SR_OP_BAR || (b >= SR_OP_BARAND && b <= SR_OP_BARPOPC); }
inline bool is_reducing_barrier(uint32_t b) { return b >= SR_OP_BARAND && b <= SR_OP_BARPOPC; }

// which operand fields an opcode reads or writes
inline bool op_writes_d(uint32_t b) {
  return (b >= SR_OP_MOV && b <= SR_OP_SNE) || b == SR_OP_S2R || b == SR_OP_LDG || b == SR_OP_LDS ||
         is_reducing_barrier(b);
}
inline bool op_reads_a(uint32_t b) {
  return (b >= SR_OP_ADD && b <= SR_OP_SNE) || b == SR_OP_LDG || b == SR_OP_STG || b == SR_OP_LDS ||
         b == SR_OP_STS || b == SR_OP_ATOMS || b == SR_OP_BRZ || b == SR_OP_BRNZ || is_reducing_barrier(b);
}
inline bool op_reads_b(uint32_t op) {
  const uint32_t b = op & 0x7Fu;
  return ((b >= SR_OP_MOV && b <= SR_OP_SNE) && !(op & SR_BIMM)) || b == SR_OP_STG || b == SR_OP_STS ||
         b == SR_OP_ATOMS;
}
inline bool is_shared_access(uint32_t b) { return b == SR_OP_LDS || b == SR_OP_STS || b == SR_OP_ATOMS; }
inline bool can_err(uint32_t b) {
  return b == SR_OP_LDS || b == SR_OP_STS || b == SR_OP_ATOMS || b == SR_OP_LDG || b == SR_OP_STG ||
         b == SR_OP_DIV || b == SR_OP_REM;
}

// Static bound for one kernel: the largest number of shared accesses and barriers a
// single thread can execute, or "unbounded" if the control-flow graph from the entry
// has a cycle.
struct KernelBound {
  bool cyclic = false;
  uint32_t accesses = 0, barriers = 0, err_pcs = 0;
  uint32_t gaccesses = 0;   // global loads and stores on the longest such path
};
// Workspace of bound_kernel: 5 arrays of ncode + 1 entries (callers own the memory).
struct BoundScratch {
  uint8_t* colour;
  uint32_t* acc;
  uint32_t* bar;
  uint32_t* stack_pc;
  uint32_t* stack_next;
  uint32_t* gacc;
};
inline KernelBound bound_kernel(const sr_instr* code, uint32_t ncode, uint32_t entry, const BoundScratch& w) {
  KernelBound kb;
  // iterative DFS with colours; longest paths by memoised post-order
  for (uint32_t i = 0; i <= ncode; ++i) { w.colour[i] = 0; w.acc[i] = 0; w.bar[i] = 0; w.gacc[i] = 0; }
  uint32_t depth = 0;
  auto succ = [&](uint32_t pc, uint32_t i, uint32_t& out) -> bool {
    if (pc >= ncode) return false;
    const uint32_t b = code[pc].op_d_a_b & 0x7Fu;
    const uint32_t t = (uint32_t)code[pc].imm;
    if (b == SR_OP_EXIT) return false;
    if (b == SR_OP_BRA) { if (i == 0) { out = t; return true; } return false; }
    if (b == SR_OP_BRZ || b == SR_OP_BRNZ) {
      if (i == 0) { out = pc + 1; return true; }
      if (i == 1) { out = t; return true; }
      return false;
    }
    if (i == 0) { out = pc + 1; return true; }
    return false;
  };
  w.stack_pc[depth] = entry;
  w.stack_next[depth] = 0;
  ++depth;
  w.colour[entry] = 1;
  while (depth) {
    const uint32_t top = depth - 1;
    uint32_t nxt;
    if (succ(w.stack_pc[top], w.stack_next[top], nxt)) {
      w.stack_next[top]++;
      if (w.colour[nxt] == 1) { kb.cyclic = true; return kb; }
      if (w.colour[nxt] == 0) {
        w.colour[nxt] = 1;
        w.stack_pc[depth] = nxt;
        w.stack_next[depth] = 0;
        ++depth;
      }
      continue;
    }
    const uint32_t pc = w.stack_pc[top];
    uint32_t a = 0, br = 0, g = 0, s;
    for (uint32_t i = 0; succ(pc, i, s); ++i) {
      a = a > w.acc[s] ? a : w.acc[s];
      br = br > w.bar[s] ? br : w.bar[s];
      g = g > w.gacc[s] ? g : w.gacc[s];
    }
    if (pc < ncode) {
      const uint32_t b = code[pc].op_d_a_b & 0x7Fu;
      a += is_shared_access(b);
      br += is_barrier(b);
      g += (b == SR_OP_LDG || b == SR_OP_STG);
      kb.err_pcs += can_err(b);
    }
    w.acc[pc] = a;
    w.bar[pc] = br;
    w.gacc[pc] = g;
    w.colour[pc] = 2;
    --depth;
  }
  kb.accesses = w.acc[entry];
  kb.barriers = w.bar[entry];
  kb.gaccesses = w.gacc[entry];
  return kb;
}

// Words of a launch's shared array that its accesses can touch: 1 + the highest in-bounds
// address of any LDS, STS or ATOMS, from intervals of the registers' values over the kernel's
// control-flow graph (thread and block indices, parameters and immediates have known ranges,
// loaded values none; a register still changing after a few visits of a loop is taken as
// unknown).  At most shmem_words, which it is when an address is unknown.
struct RangeScratch {
  struct State {
    int32_t lo[16], hi[16];
    uint32_t visits;             // 0: not reached
    uint32_t by_params;          // registers whose interval follows from the launch's parameters
  };
  std::vector<int32_t> leader;   // per pc: index of its state, -1 inside a straight line
  std::vector<State> states;
  std::vector<uint8_t> queued;
  bool by_params = false;        // the last result follows from the parameters (some address's interval does)
  // the last results for the program at hand (shared_reach_of)
  struct Seen {
    uint32_t entry, block_dim, grid, block_begin, block_count, shmem_words, nparams;
    int32_t params[4];
    bool by_params;
    uint32_t reach;
  };
  std::vector<Seen> seen;
  uint64_t analyses = 0;
};
inline uint32_t shared_reach(const sr_instr* code, uint32_t ncode, uint32_t entry, const sr_launch& L, RangeScratch& w) {
  const uint32_t shw = L.shmem_words;
  w.by_params = false;
  if (!shw) return 0;
  ++w.analyses;
  using State = RangeScratch::State;
  // leaders: the entry, branch targets and what follows a branch
  w.leader.assign(ncode + 1, -1);
  w.states.clear();
  auto lead = [&](uint32_t pc) {
    if (pc < ncode && w.leader[pc] < 0) {
      w.leader[pc] = (int32_t)w.states.size();
      w.states.push_back(State{});
    }
  };
  lead(entry);
  for (uint32_t pc = 0; pc < ncode; ++pc) {
    const uint32_t b = code[pc].op_d_a_b & 0x7Fu;
    if (b == SR_OP_BRA || b == SR_OP_BRZ || b == SR_OP_BRNZ) {
      lead((uint32_t)code[pc].imm);
      lead(pc + 1);
    }
  }
  w.queued.assign(ncode + 1, 0);
  uint32_t reach = 0, next = ncode;              // next: the lowest queued leader
  auto flow = [&](const State& s, uint32_t pc) { // join s into the leader at pc
    if (pc >= ncode) return;
    State& t = w.states[(size_t)w.leader[pc]];
    bool changed = t.visits == 0;
    for (uint32_t r = 0; r < 16; ++r) {
      const int32_t lo = t.visits ? std::min(t.lo[r], s.lo[r]) : s.lo[r];
      const int32_t hi = t.visits ? std::max(t.hi[r], s.hi[r]) : s.hi[r];
      if (t.visits && (lo != t.lo[r] || hi != t.hi[r])) {
        changed = true;
        if (t.visits > 4) {                      // still changing: unknown
          t.lo[r] = INT32_MIN;
          t.hi[r] = INT32_MAX;
          continue;
        }
      }
      t.lo[r] = lo;
      t.hi[r] = hi;
    }
    const bool more = (s.by_params & ~t.by_params) != 0;
    t.by_params |= s.by_params;
    t.visits += changed;
    if (changed || more) {
      w.queued[pc] = 1;
      next = std::min(next, pc);
    }
  };
  State s{};
  for (uint32_t q = 0; q < 4 && q < L.nparams; ++q) {
    s.lo[q] = s.hi[q] = L.params[q];
    s.by_params |= 1u << q;
  }
  flow(s, entry);
  const int64_t first = L.block_begin, blocks = L.block_count ? L.block_count : L.grid;
  while (next < ncode) {
    uint32_t pc = next;
    w.queued[pc] = 0;
    s = w.states[(size_t)w.leader[pc]];
    next = ncode;
    for (uint32_t i = pc + 1; i < ncode; ++i)
      if (w.queued[i]) {
        next = i;
        break;
      }
    for (;;) {                                   // to the end of the straight line
      const uint32_t word = code[pc].op_d_a_b, op = word & 0xFFu, b = op & 0x7Fu;
      const uint32_t d = (word >> 8) & 0xFFu, ra = (word >> 16) & 0xFFu, rb = (word >> 24) & 0xFFu;
      const int64_t imm = code[pc].imm;
      const bool za = ra == SR_RZ || ra > 15, zb = rb == SR_RZ || rb > 15;
      const int64_t al = za ? 0 : s.lo[ra], ah = za ? 0 : s.hi[ra];
      int64_t bl = zb ? 0 : s.lo[rb], bh = zb ? 0 : s.hi[rb];
      if (op & SR_BIMM) bl = bh = imm;
      int64_t lo = INT32_MIN, hi = INT32_MAX;    // the result's interval (unknown)
      const bool pa = !za && ((s.by_params >> ra) & 1u), pb = !(op & SR_BIMM) && !zb && ((s.by_params >> rb) & 1u);
      switch (b) {
        case SR_OP_MOV: lo = bl; hi = bh; break;
        case SR_OP_ADD: lo = al + bl; hi = ah + bh; break;
        case SR_OP_SUB: lo = al - bh; hi = ah - bl; break;
        case SR_OP_MUL: {
          const int64_t x[4] = {al * bl, al * bh, ah * bl, ah * bh};
          lo = *std::min_element(x, x + 4);
          hi = *std::max_element(x, x + 4);
          break;
        }
        case SR_OP_DIV:
          if (bl == bh && bl > 0) { lo = al / bl; hi = ah / bl; }
          break;
        case SR_OP_REM:
          if (bl == bh && bl > 0) {
            lo = al < 0 ? -(bl - 1) : 0;
            hi = ah > 0 ? std::min(ah, bl - 1) : 0;
          }
          break;
        case SR_OP_AND:
          if (bl >= 0 || al >= 0) {
            lo = 0;
            hi = bl < 0 ? ah : al < 0 ? bh : std::min(ah, bh);
          }
          break;
        case SR_OP_OR:
        case SR_OP_XOR:
          if (al >= 0 && bl >= 0) {
            int64_t m = 1;
            while (m <= ah || m <= bh) m <<= 1;
            lo = 0;
            hi = m - 1;
          }
          break;
        case SR_OP_SHL:
          if (bl == bh) { lo = al * ((int64_t)1 << (bl & 31)); hi = ah * ((int64_t)1 << (bl & 31)); }
          break;
        case SR_OP_SHR:
          if (bl == bh) { lo = al >> (bl & 31); hi = ah >> (bl & 31); }
          break;
        case SR_OP_MIN: lo = std::min(al, bl); hi = std::min(ah, bh); break;
        case SR_OP_MAX: lo = std::max(al, bl); hi = std::max(ah, bh); break;
        case SR_OP_SLT: case SR_OP_SLE: case SR_OP_SEQ: case SR_OP_SNE: case SR_OP_BARAND: case SR_OP_BAROR:
          lo = 0; hi = 1;
          break;
        case SR_OP_BARPOPC: lo = 0; hi = L.block_dim; break;
        case SR_OP_S2R:
          if (imm == SR_SREG_TID) { lo = 0; hi = (int64_t)L.block_dim - 1; }
          else if (imm == SR_SREG_BID) { lo = first; hi = first + blocks - 1; }
          else if (imm == SR_SREG_BDIM) lo = hi = L.block_dim;
          else if (imm == SR_SREG_GDIM) lo = hi = L.grid;
          else lo = hi = 32;
          break;
        case SR_OP_LDS: case SR_OP_STS: case SR_OP_ATOMS: {
          const int64_t l = al + imm, h = ah + imm;
          w.by_params = w.by_params || pa;
          if (l < INT32_MIN || h > INT32_MAX) reach = shw;
          else if (h >= 0 && l < (int64_t)shw) reach = std::max(reach, (uint32_t)std::min<int64_t>(h + 1, shw));
          break;
        }
        default: break;
      }
      if (op_writes_d(b) && d < 16) {
        const bool fits = lo >= INT32_MIN && hi <= INT32_MAX;
        s.lo[d] = fits ? (int32_t)lo : INT32_MIN;
        s.hi[d] = fits ? (int32_t)hi : INT32_MAX;
        // (comparisons and what is loaded, read or counted: the same interval for any parameters)
        const bool from = b == SR_OP_MOV ? pb : b >= SR_OP_ADD && b <= SR_OP_MAX && (pa || pb);
        s.by_params = (s.by_params & ~(1u << d)) | (from ? 1u << d : 0u);
      }
      if (reach == shw || b == SR_OP_EXIT) break;
      if (b == SR_OP_BRA || b == SR_OP_BRZ || b == SR_OP_BRNZ) {
        flow(s, (uint32_t)code[pc].imm);
        if (b != SR_OP_BRA) flow(s, pc + 1);
        break;
      }
      if (++pc >= ncode) break;
      if (w.leader[pc] >= 0) {
        flow(s, pc);
        break;
      }
    }
    if (reach == shw) break;
  }
  return reach;
}

// The same for a program's launches one after the other (w.seen is empty before the first): the analysis
// (11 us for a kernel of 3,000 instructions) runs once for launches of the same shape
// whose addresses do not follow from the parameters, or with the same parameters.
inline uint32_t shared_reach_of(const sr_instr* code, uint32_t ncode, uint32_t entry, const sr_launch& L, RangeScratch& w) {
  RangeScratch::Seen k{entry, L.block_dim, L.grid, L.block_begin, L.block_count, L.shmem_words, L.nparams, {}, false, 0};
  for (uint32_t q = 0; q < 4 && q < L.nparams; ++q) k.params[q] = L.params[q];
  for (size_t i = w.seen.size(); i-- > 0;) {
    const RangeScratch::Seen& o = w.seen[i];
    if (o.entry == k.entry && o.block_dim == k.block_dim && o.grid == k.grid && o.block_begin == k.block_begin &&
        o.block_count == k.block_count && o.shmem_words == k.shmem_words && o.nparams == k.nparams &&
        (!o.by_params || std::equal(k.params, k.params + 4, o.params)))
      return o.reach;
  }
  k.reach = shared_reach(code, ncode, entry, L, w);
  k.by_params = w.by_params;
  if (w.seen.size() >= 16) w.seen.erase(w.seen.begin());
  w.seen.push_back(k);
  return k.reach;
}

inline int validate(const sr_program* p, char* msg, size_t len) {
  auto bad = [&](const char* fmt, uint32_t x, uint32_t y) {
    if (msg && len) snprintf(msg, len, fmt, x, y);
    return SR_E_INVAL;
  };
  if (!p || !p->code || p->ncode == 0 || p->ncode > SR_MAX_CODE) return bad("code size %u outside 1..%u", p ? p->ncode : 0, SR_MAX_CODE);
  if (!p->kernel_entry || p->nkernels == 0) return bad("no kernels (%u, %u)", 0, 0);
  for (uint32_t k = 0; k < p->nkernels; ++k)
    if (p->kernel_entry[k] >= p->ncode) return bad("kernel %u entry %u out of range", k, p->kernel_entry[k]);
  for (uint32_t pc = 0; pc < p->ncode; ++pc) {
    const uint32_t w = p->code[pc].op_d_a_b, op = w & 0xFFu, b = op & 0x7Fu;
    const uint32_t d = (w >> 8) & 0xFFu, ra = (w >> 16) & 0xFFu, rb = (w >> 24) & 0xFFu;
    const int32_t imm = p->code[pc].imm;
    const bool alu = b >= SR_OP_MOV && b <= SR_OP_SNE;
    if (b < SR_OP_MOV || b > SR_OP_BARPOPC || (op & 0x40u) || ((op & SR_BIMM) && !alu))
      return bad("pc %u: bad opcode 0x%x", pc, op);
    auto reg_ok = [](uint32_t r) { return r < 16 || r == SR_RZ; };
    if ((op_writes_d(b) && !reg_ok(d)) || (op_reads_a(b) && !reg_ok(ra)) || (op_reads_b(op) && !reg_ok(rb)))
      return bad("pc %u: bad register field (op %u)", pc, b);
    if ((b == SR_OP_BRA || b == SR_OP_BRZ || b == SR_OP_BRNZ) && (imm < 0 || (uint32_t)imm > p->ncode))
      return bad("pc %u: branch target %u out of range", pc, (uint32_t)imm);
    if (b == SR_OP_S2R && (imm < 0 || imm > SR_SREG_WARPSIZE)) return bad("pc %u: bad special register %u", pc, (uint32_t)imm);
  }
  if (p->nlaunches && !p->launches) return bad("launch table missing (%u launches)", p->nlaunches, 0);
  for (uint32_t l = 0; l < p->nlaunches; ++l) {
    const sr_launch& L = p->launches[l];
    if (L.kernel >= p->nkernels) return bad("launch %u: kernel %u out of range", l, L.kernel);
    if (L.grid == 0 || L.grid > (1u << 30)) return bad("launch %u: grid %u", l, L.grid);
    if (L.block_dim == 0 || L.block_dim > SR_MAX_BLOCK_DIM) return bad("launch %u: block_dim %u", l, L.block_dim);
    if (L.shmem_words > SR_MAX_SHMEM_WORDS) return bad("launch %u: shmem_words %u", l, L.shmem_words);
    if (L.nparams > 4) return bad("launch %u: nparams %u", l, L.nparams);
    if (L.wait > l) return bad("launch %u: waits for launch %u, which is not an earlier one", l, L.wait - 1);
    if ((L.block_count == 0 && L.block_begin != 0) || (uint64_t)L.block_begin + L.block_count > L.grid)
      return bad("launch %u: block range starting at %u outside the grid", l, L.block_begin);
  }
  if (p->global_words >= (1ull << 31)) return bad("global arena too large (%u)", (uint32_t)(p->global_words >> 20), 0);
  if (p->global_words && !p->global_init) return bad("global_init missing (%u words)", (uint32_t)p->global_words, 0);
  return SR_OK;
}

// Register renaming of one program: the registers it touches (plus the parameter
// registers r0..r(maxp-1)) become rows 0..n-1 in ascending order, the zero row is n.
struct RegMap {
  uint8_t row[256];
  uint32_t nrows;
};
inline RegMap map_registers(const sr_program& P) {
  bool used[16] = {};
  uint32_t maxp = 0;
  for (uint32_t l = 0; l < P.nlaunches; ++l) maxp = std::max(maxp, P.launches[l].nparams);
  for (uint32_t r = 0; r < maxp; ++r) used[r] = true;
  for (uint32_t pc = 0; pc < P.ncode; ++pc) {
    const uint32_t w = P.code[pc].op_d_a_b, op = w & 0xFFu, b = op & 0x7Fu;
    const uint32_t d = (w >> 8) & 0xFFu, ra = (w >> 16) & 0xFFu, rb = (w >> 24) & 0xFFu;
    if (op_writes_d(b) && d < 16) used[d] = true;
    if (op_reads_a(b) && ra < 16) used[ra] = true;
    if (op_reads_b(op) && rb < 16) used[rb] = true;
  }
  RegMap m;
  uint32_t n = 0;
  for (uint32_t r = 0; r < 16; ++r) m.row[r] = used[r] ? (uint8_t)n++ : 0;
  m.nrows = n + 1;
  return m;
}

// pack one instruction: sources that are RZ or unused read the zero row; destinations
// that are RZ or absent become kNoDest
inline uint2 pack(const sr_instr& in, const RegMap& m) {
  const uint32_t w = in.op_d_a_b, op = w & 0xFFu, b = op & 0x7Fu;
  const bool bimm = (op & SR_BIMM) != 0;
  uint32_t d = (w >> 8) & 0xFFu, ra = (w >> 16) & 0xFFu, rb = (w >> 24) & 0xFFu, imm = (uint32_t)in.imm, form;
  const uint32_t zrow = m.nrows - 1;
  d = (op_writes_d(b) && d != SR_RZ) ? m.row[d] : sr::kNoDest;
  ra = (op_reads_a(b) && ra != SR_RZ) ? m.row[ra] : zrow;
  rb = (op_reads_b(op) && rb != SR_RZ) ? m.row[rb] : zrow;
  auto of = [&](uint32_t f) { return bimm ? f : f + 1u; };
  switch (b) {
    case SR_OP_MOV:                              // (of a register: a plus the zero row)
      form = bimm ? sr::F_MOVI : sr::F_MOVR;
      ra = bimm ? zrow : rb;
      rb = zrow;
      break;
    case SR_OP_ADD: form = bimm ? sr::F_ADDI : sr::F_ADDR; break;
    case SR_OP_SUB:
      form = bimm ? sr::F_ADDI : sr::F_SUBR;
      if (bimm) imm = 0u - imm;
      break;
    case SR_OP_MUL: form = bimm ? sr::F_MULI : sr::F_MULR; break;
    case SR_OP_SHL:
      form = bimm ? sr::F_MULI : sr::F_SHL + 1u;
      if (bimm) imm = 1u << (imm & 31u);
      break;
    case SR_OP_AND: form = of(sr::F_AND); break;
    case SR_OP_OR: form = of(sr::F_OR); break;
    case SR_OP_XOR: form = of(sr::F_XOR); break;
    case SR_OP_SHR: form = of(sr::F_SHR); break;
    case SR_OP_MIN: form = of(sr::F_MIN); break;
    case SR_OP_MAX: form = of(sr::F_MAX); break;
    case SR_OP_SLT: form = of(sr::F_SLT); break;
    case SR_OP_SLE: form = of(sr::F_SLE); break;
    case SR_OP_SEQ: form = of(sr::F_SEQ); break;
    case SR_OP_SNE: form = of(sr::F_SNE); break;
    case SR_OP_DIV: form = bimm ? sr::F_DIVI : sr::F_DIVR; break;
    case SR_OP_REM: form = bimm ? sr::F_REMI : sr::F_REMR; break;
    case SR_OP_S2R: form = sr::F_S2R; break;
    case SR_OP_LDG: form = sr::F_LDG; break;
    case SR_OP_STG: form = sr::F_STG; break;
    case SR_OP_LDS: form = sr::F_LDS; break;
    case SR_OP_STS: form = sr::F_STS; break;
    case SR_OP_ATOMS: form = sr::F_ATOMS; break;
    case SR_OP_BRA: form = sr::F_BRA; break;
    case SR_OP_BRZ: form = sr::F_BRZ; break;
    case SR_OP_BRNZ: form = sr::F_BRNZ; break;
    case SR_OP_BAR: form = sr::F_BAR; break;
    case SR_OP_BARAND: form = sr::F_BARAND; break;
    case SR_OP_BAROR: form = sr::F_BAROR; break;
    case SR_OP_BARPOPC: form = sr::F_BARPOPC; break;
    default: form = sr::F_EXIT; break;
  }
  return make_uint2(sr::pk_make(form, d, ra, rb), imm);
}

// The EXIT sentinel after a program's last instruction (running past the end exits).
inline uint2 exit_sentinel(const RegMap& m) {
  return make_uint2(sr::pk_make(sr::F_EXIT, sr::kNoDest, m.nrows - 1, m.nrows - 1), 0);
}

// Marks, chains and run lengths (sr_internal.h) of n packed instructions; run: one byte each;
// target[pc]: a branch or an entry may lead there.  A run holds straight-line successors only and
// no branch, so its length is right from any entry pc.  The interpreter ignores the operand mark of
// the first instruction it executes of a run and the result mark of the last one, so the marks
// hold wherever a run is entered or cut: a value is kept back only while the instructions up to
// its overwriting follow in the same straight line.  Runs are cut between chains, and nothing
// leads into a chain's middle, so no thread ever stands there (but for one whose block is out of
// rounds, and stops).
inline void set_runs(uint2* code, uint8_t* run, uint32_t n, const uint8_t* target) {
  auto runs = [&](uint32_t pc) { return sr::pk_form(code[pc].x) < sr::F_LDS; };
  uint32_t live = 0;                             // rows read later, or alive past the run
  for (uint32_t pc = n; pc-- > 0;) {
    if (!runs(pc)) continue;
    uint32_t x = code[pc].x;
    const uint32_t form = sr::pk_form(x), d = sr::pk_d(x);
    uint32_t a = sr::pk_a(x), b = sr::pk_b(x);
    if (pc + 1 >= n || !runs(pc + 1)) live = ~0u;   // (the last of its run)
    if (d != sr::kNoDest) {
      if (!((live >> d) & 1u)) x |= sr::kDeadD;
      live &= ~(1u << d);
    }
    // the previous instruction's result as operand a, swapped there where the operation allows
    const uint32_t before = pc && runs(pc - 1) ? sr::pk_d(code[pc - 1].x) : sr::kNoDest;
    const bool commutes = form == sr::F_ADDR || form == sr::F_MULR || form == sr::F_AND + 1u || form == sr::F_OR + 1u ||
                          form == sr::F_XOR + 1u || form == sr::F_MIN + 1u || form == sr::F_MAX + 1u ||
                          form == sr::F_SEQ + 1u || form == sr::F_SNE + 1u;
    if (commutes && b == before && a != before) std::swap(a, b);
    if (form == sr::F_MOVI || (a == before && before != sr::kNoDest))
      x |= sr::kFwdA;                            // (MOVI: no operand a to load)
    else
      live |= 1u << a;
    if (!sr::pk_imm(form)) live |= 1u << b;
    if (form <= sr::F_MULI) b = 1;               // (a chain of one)
    code[pc].x = (x & 0xFFFFu) | a << 16 | b << 24;
  }
  for (uint32_t pc = 0; pc < n;) {               // chains
    uint32_t len = 1;
    if (sr::pk_form(code[pc].x) <= sr::F_MULI) {
      uint32_t last = code[pc].x;
      while (len < sr::kRunMax && pc + len < n && !target[pc + len] && (last & sr::kDeadD)) {
        uint2& e = code[pc + len];
        if (sr::pk_form(e.x) > sr::F_MULI || !(e.x & sr::kFwdA)) break;
        last = e.x;
        const uint32_t form = sr::pk_form(e.x);
        e = form == sr::F_MULI ? make_uint2(e.y, 0u) : make_uint2(form, e.y);   // (MOVI 0, ADDI 1)
        ++len;
      }
      code[pc].x = (code[pc].x & ~(0xFF000000u | 0xFF00u | sr::kDeadD)) | (last & (0xFF00u | sr::kDeadD)) | len << 24;
    }
    run[pc] = (uint8_t)len;
    for (uint32_t i = 1; i < len; ++i) run[pc + i] = 0;
    pc += len;
  }
  // from the lengths of single instructions and chains, those of runs (never past kRunMax)
  uint32_t next = 0;                             // the run length after this place
  for (uint32_t pc = n; pc-- > 0;) {
    if (!run[pc]) continue;                      // (inside a chain)
    const uint32_t len = run[pc];
    if (!runs(pc)) {
      run[pc] = 0;
      next = 0;
      continue;
    }
    next = len + next <= sr::kRunMax ? len + next : len;
    run[pc] = (uint8_t)next;
  }
}

// A program as it is staged: out holds packed_words(ncode) pairs.
inline uint32_t packed_words(uint32_t ncode) { return sr::packed_bytes(ncode) / 8u; }
inline void pack_program(const sr_program& P, const RegMap& m, uint2* out) {
  const uint32_t n = P.ncode + 1;
  uint8_t target[SR_MAX_CODE + 1] = {};
  for (uint32_t pc = 0; pc < P.ncode; ++pc) {
    out[pc] = pack(P.code[pc], m);
    const uint32_t b = P.code[pc].op_d_a_b & 0x7Fu;
    if (b == SR_OP_BRA || b == SR_OP_BRZ || b == SR_OP_BRNZ) target[(uint32_t)P.code[pc].imm] = 1;
  }
  for (uint32_t k = 0; k < P.nkernels; ++k) target[P.kernel_entry[k]] = 1;
  for (uint32_t i = P.ncode; i < packed_words(P.ncode); ++i) out[i] = make_uint2(0u, 0u);
  for (uint32_t i = P.ncode; i < sr::ir_code_bytes(P.ncode) / 8u; ++i) out[i] = exit_sentinel(m);
  set_runs(out, reinterpret_cast<uint8_t*>(out) + sr::ir_code_bytes(P.ncode), n, target);
}

inline uint32_t key_bits_for(uint32_t shw) {
  uint32_t b = 1;
  while ((1u << b) < shw) ++b;
  return b;
}


// The launches (indices within the program, or `none`) that launch l follows: the previous
// launch of its stream and the launch it waits for (Sec. 3, streams and events).
inline void launch_deps(const sr_launch* launches, uint32_t l, uint32_t none, uint32_t& prev, uint32_t& wait) {
  prev = none;
  for (uint32_t m = l; m-- > 0;)
    if (launches[m].stream == launches[l].stream) {
      prev = m;
      break;
    }
  wait = launches[l].wait ? launches[l].wait - 1 : none;
}

// Access-log region (records per block, even) of one launch: the static bound of its
// kernel, or `loop_records` for kernels with loops, plus room for barrier/error records.
inline uint64_t launch_log_cap(const KernelBound& k, uint32_t block_dim, uint32_t check_races, uint32_t loop_records) {
  uint64_t recs, misc;
  if (k.cyclic) {
    recs = loop_records;
    misc = 4ull * (1 + k.err_pcs) > 256 ? 4ull * (1 + k.err_pcs) : 256;
  } else {
    recs = (uint64_t)k.accesses * block_dim;
    misc = (uint64_t)(k.barriers + 1) * (1 + k.err_pcs) + 1;
  }
  if (!check_races) recs = 0;
  return (recs + 2 * misc + 1) & ~1ull;
}

// Global-log region (records per block, even) of one launch for the global-memory race
// check: the kernel's static bound of global loads and stores per thread, or `loop_records`
// for kernels with loops.
inline uint64_t launch_glog_cap(const KernelBound& k, uint32_t block_dim, uint32_t loop_records) {
  const uint64_t recs = k.cyclic ? (uint64_t)loop_records : (uint64_t)k.gaccesses * block_dim;
  return (recs + 1) & ~1ull;
}

// Launch-order bit matrix of one program (Sec. 3, streams and events): bit l * nl + m is set
// when launch m precedes launch l through stream order and event waits, transitively.
// Returns false (nothing written) when every pair of launches is ordered.
inline bool launch_order_bits(const sr_launch* launches, uint32_t nl, std::vector<uint32_t>& bits) {
  std::vector<uint8_t> before((size_t)nl * nl, 0);
  for (uint32_t l = 0; l < nl; ++l) {
    uint32_t prev, wait;
    launch_deps(launches, l, UINT32_MAX, prev, wait);
    for (uint32_t d : {prev, wait}) {
      if (d == UINT32_MAX) continue;
      before[(size_t)l * nl + d] = 1;
      for (uint32_t m = 0; m < nl; ++m)
        if (before[(size_t)d * nl + m]) before[(size_t)l * nl + m] = 1;
    }
  }
  bool all = true;
  for (uint32_t l = 0; l < nl && all; ++l)
    for (uint32_t m = 0; m < l; ++m)
      if (!before[(size_t)l * nl + m]) { all = false; break; }
  if (all) return false;
  bits.assign(((size_t)nl * nl + 31) / 32, 0u);
  for (size_t i = 0; i < (size_t)nl * nl; ++i)
    if (before[i]) bits[i / 32] |= 1u << (i % 32);
  return true;
}

}  // namespace host
}  // namespace sr
