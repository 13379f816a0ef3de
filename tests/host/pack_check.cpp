// Host check of the packed instruction forms: random programs, every run of instructions executed
// the way the interpreter does (forms, chains, forwarded operands, dead results) against the plain
// code.  Prints "ok <instructions> <chained>" or the first difference.
#include <cstdio>
#include <random>
#include <vector>

#include "host_prep.h"

using namespace sr;
using namespace sr::host;

static int32_t alu(uint32_t op, int32_t x, int32_t y) {
  const uint32_t a = (uint32_t)x, b = (uint32_t)y;
  switch (op) {
    case SR_OP_MOV: return y;
    case SR_OP_ADD: return (int32_t)(a + b);
    case SR_OP_SUB: return (int32_t)(a - b);
    case SR_OP_MUL: return (int32_t)(a * b);
    case SR_OP_AND: return (int32_t)(a & b);
    case SR_OP_OR: return (int32_t)(a | b);
    case SR_OP_XOR: return (int32_t)(a ^ b);
    case SR_OP_SHL: return (int32_t)(a << (b & 31));
    case SR_OP_SHR: return x >> (b & 31);
    case SR_OP_MIN: return std::min(x, y);
    case SR_OP_MAX: return std::max(x, y);
    case SR_OP_SLT: return x < y;
    case SR_OP_SLE: return x <= y;
    case SR_OP_SEQ: return x == y;
    default: return x != y;
  }
}

int main() {
  const uint32_t ops[15] = {SR_OP_MOV, SR_OP_ADD, SR_OP_SUB, SR_OP_MUL, SR_OP_AND, SR_OP_OR,  SR_OP_XOR, SR_OP_SHL,
                            SR_OP_SHR, SR_OP_MIN, SR_OP_MAX, SR_OP_SLT, SR_OP_SLE, SR_OP_SEQ, SR_OP_SNE};
  const uint32_t forms[11] = {SR_OP_AND, SR_OP_OR,  SR_OP_XOR, SR_OP_SHL, SR_OP_SHR, SR_OP_MIN,
                              SR_OP_MAX, SR_OP_SLT, SR_OP_SLE, SR_OP_SEQ, SR_OP_SNE};   // from form 8, two each
  std::mt19937 g(1);
  long total = 0, chained = 0;
  for (int it = 0; it < 4000; ++it) {
    const uint32_t n = it % 3 ? 1 + g() % 30 : 1 + g() % 400;
    const int mode = (int)(g() % 4);             // 0: all operations; else mostly chains, 1: without branches
    std::vector<sr_instr> code(n);
    std::vector<uint32_t> starts = {0};
    for (uint32_t i = 0; i < n; ++i) {
      uint32_t op = mode ? (g() % 2 ? SR_OP_ADD : SR_OP_MUL) : ops[g() % 15];
      if (mode == 2 && g() % 8 == 0) op = SR_OP_MOV;
      const uint32_t nr = mode == 1 ? 2 : mode == 3 ? 1 : 5;
      auto reg = [&]() { return mode != 1 && g() % 20 == 0 ? 255u : (uint32_t)(g() % nr); };
      const uint32_t d = reg(), a = reg(), b = reg();
      int32_t im = (int32_t)g();
      if (g() % 2) im %= 40;
      uint32_t w = op | (mode == 1 || g() % 4 ? 0x80u : 0u) | d << 8 | a << 16 | b << 24;
      if (mode != 1 && g() % 12 == 0) {
        w = SR_OP_BRZ | 255u << 16;
        im = (int32_t)(g() % (n + 1));
        starts.push_back((uint32_t)im);
        starts.push_back(i + 1);
      }
      code[i] = {w, im};
    }
    sr_launch L{};
    L.nparams = 2;
    L.grid = 1;
    L.block_dim = 32;
    uint32_t entry = 0;
    sr_program P{};
    P.code = code.data();
    P.ncode = n;
    P.kernel_entry = &entry;
    P.nkernels = 1;
    P.launches = &L;
    P.nlaunches = 1;
    const RegMap m = map_registers(P);
    std::vector<uint2> out(packed_words(n));
    pack_program(P, m, out.data());
    const uint8_t* run = reinterpret_cast<const uint8_t*>(out.data()) + ir_code_bytes(n);
    bool used[16] = {true, true};
    for (const sr_instr& c : code) {
      const uint32_t w = c.op_d_a_b, op = w & 255u, base = op & 127u;
      auto use = [&](uint32_t r) { if (r < 16) used[r] = true; };
      if (op_writes_d(base)) use((w >> 8) & 255u);
      if (op_reads_a(base)) use((w >> 16) & 255u);
      if (op_reads_b(op)) use(w >> 24);
    }
    for (uint32_t start : starts) {
      if (start >= n || pk_form(out[start].x) >= F_LDS) continue;
      int32_t R[16];                             // plain registers; F: the rows
      std::vector<int32_t> F(m.nrows, 0);
      for (int r = 0; r < 16; ++r) {
        R[r] = (int32_t)g();
        if (used[r]) F[m.row[r]] = R[r];
      }
      for (uint32_t pc = start; pc < n && pk_form(out[pc].x) < F_LDS;) {
        const uint32_t len = run[pc];
        if (!len || pc + len > n) return printf("run of %u at %u\n", len, pc), 1;
        for (uint32_t i = pc; i < pc + len; ++i) {
          const uint32_t w = code[i].op_d_a_b, op = w & 255u, a = (w >> 16) & 255u, b = w >> 24, d = (w >> 8) & 255u;
          const int32_t r = alu(op & 127u, a < 16 ? R[a] : 0, op & 0x80u ? code[i].imm : b < 16 ? R[b] : 0);
          if (d < 16) R[d] = r;
        }
        int32_t c = 0x5a5a5a5a;                  // the previous result
        uint32_t keep = 0;
        for (uint32_t q = pc; q < pc + len;) {
          const uint32_t x = out[q].x, y = out[q].y, f = pk_form(x);
          if (!(x & keep)) c = F[pk_a(x)];
          if (f <= F_MULI) {
            const uint32_t count = pk_b(x);
            c = (int32_t)((uint32_t)c * (f == F_MULI ? y : f) + (f == F_MULI ? 0u : y));
            for (uint32_t e = 1; e < count; ++e, ++chained) c = (int32_t)((uint32_t)c * out[q + e].x + out[q + e].y);
            q += count;
            if (q > pc + len) return printf("chain past its run at %u\n", pc), 1;
          } else {
            const int32_t b = pk_imm(f) ? (int32_t)y : F[pk_b(x)];
            c = f == F_MOVR || f == F_ADDR ? (int32_t)((uint32_t)c + (uint32_t)b)
                : f == F_SUBR              ? (int32_t)((uint32_t)c - (uint32_t)b)
                : f == F_MULR              ? (int32_t)((uint32_t)c * (uint32_t)b)
                                           : alu(forms[(f - 8) / 2], c, b);
            ++q;
          }
          keep = kFwdA;
          if ((q >= pc + len || !(x & kDeadD)) && pk_d(x) != kNoDest) F[pk_d(x)] = c;
          ++total;
        }
        pc += len;
        if (pc >= n || pk_form(out[pc].x) >= F_LDS)   // (cut runs leave only what they overwrite)
          for (int r = 0; r < 16; ++r)
            if (used[r] && F[m.row[r]] != R[r]) return printf("program %d from %u: register %d\n", it, start, r), 1;
      }
    }
  }
  printf("ok %ld %ld\n", total, chained);
  return 0;
}
