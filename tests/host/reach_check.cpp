// Host check of shared_reach: random kernels run thread by thread with arbitrary loaded values; no
// shared access that is in bounds lies past the words the analysis gives.  Prints "ok <accesses>
// <kernels whose reach is below their array>" or the first access outside.
#include <cstdio>
#include <random>
#include <vector>

#include "host_prep.h"

using namespace sr;
using namespace sr::host;

int main() {
  const uint32_t alu[17] = {SR_OP_MOV, SR_OP_ADD, SR_OP_SUB, SR_OP_MUL, SR_OP_DIV, SR_OP_REM, SR_OP_AND, SR_OP_OR, SR_OP_XOR,
                            SR_OP_SHL, SR_OP_SHR, SR_OP_MIN, SR_OP_MAX, SR_OP_SLT, SR_OP_SLE, SR_OP_SEQ, SR_OP_SNE};
  std::mt19937 g(7);
  RangeScratch scratch;
  long accesses = 0, below = 0;
  for (int it = 0; it < 6000; ++it) {
    const uint32_t n = 4 + g() % 40, shw = 1 + g() % 3000;
    std::vector<sr_instr> code(n);
    auto reg = [&]() { return g() % 16 == 0 ? (uint32_t)SR_RZ : (uint32_t)(g() % 6); };
    for (uint32_t i = 0; i < n; ++i) {
      const uint32_t d = reg(), a = reg(), b = reg(), what = g() % 16;
      int32_t im = (int32_t)(g() % 80) - 16;
      if (g() % 20 == 0) im = (int32_t)g();
      uint32_t op;
      if (what < 9) {
        op = alu[g() % 17] | (g() % 2 ? SR_BIMM : 0u);
        if (g() % 3 == 0) op = SR_OP_AND | SR_BIMM;
      } else if (what < 11) {
        op = g() % 3 ? SR_OP_STS : SR_OP_ATOMS;
      } else if (what == 11) {
        op = SR_OP_LDS;
      } else if (what == 12) {
        op = g() % 2 ? SR_OP_LDG : SR_OP_S2R;
        if (op == SR_OP_S2R) im = (int32_t)(g() % 5);
      } else if (what == 13) {
        op = g() % 3 == 0 ? SR_OP_BARPOPC : g() % 2 ? SR_OP_BAROR : SR_OP_BARAND;
      } else {
        op = g() % 5 == 0 ? SR_OP_BRA : g() % 2 ? SR_OP_BRZ : SR_OP_BRNZ;
        im = (int32_t)(g() % (n + 1));
      }
      code[i] = {op | d << 8 | a << 16 | b << 24, im};
    }
    sr_launch L{};
    L.grid = 1 + g() % 50;
    L.block_dim = 1 + g() % 1024;
    L.shmem_words = shw;
    L.nparams = g() % 3;
    for (uint32_t q = 0; q < L.nparams; ++q) L.params[q] = (int32_t)(g() % 200) - 50;
    if (g() % 3 == 0) {
      L.block_begin = g() % L.grid;
      L.block_count = 1 + g() % (L.grid - L.block_begin);
    }
    const uint32_t reach = shared_reach(code.data(), n, 0, L, scratch);
    if (reach > shw) return printf("kernel %d: reach %u of %u words\n", it, reach, shw), 1;
    below += reach < shw;
    const uint32_t first = L.block_begin, blocks = L.block_count ? L.block_count : L.grid;
    for (int run = 0; run < 12; ++run) {
      const int32_t tid = run == 0 ? 0 : run == 1 ? (int32_t)L.block_dim - 1 : (int32_t)(g() % L.block_dim);
      int32_t R[6] = {};
      for (uint32_t q = 0; q < L.nparams; ++q) R[q] = L.params[q];
      uint32_t pc = 0;
      for (int step = 0; step < 400 && pc < n; ++step) {
        const uint32_t w = code[pc].op_d_a_b, op = w & 255u, base = op & 127u, d = (w >> 8) & 255u;
        const int32_t im = code[pc].imm, x = ((w >> 16) & 255u) < 6 ? R[(w >> 16) & 255u] : 0;
        const int32_t y = op & SR_BIMM ? im : (w >> 24) < 6 ? R[w >> 24] : 0;
        const uint32_t a = (uint32_t)x, b = (uint32_t)y;
        int32_t r = 0;
        uint32_t next = pc + 1;
        switch (base) {
          case SR_OP_MOV: r = y; break;
          case SR_OP_ADD: r = (int32_t)(a + b); break;
          case SR_OP_SUB: r = (int32_t)(a - b); break;
          case SR_OP_MUL: r = (int32_t)(a * b); break;
          case SR_OP_DIV: r = y == 0 ? 0 : y == -1 ? (int32_t)(0u - a) : x / y; break;
          case SR_OP_REM: r = y == 0 || y == -1 ? 0 : x % y; break;
          case SR_OP_AND: r = x & y; break;
          case SR_OP_OR: r = x | y; break;
          case SR_OP_XOR: r = x ^ y; break;
          case SR_OP_SHL: r = (int32_t)(a << (b & 31)); break;
          case SR_OP_SHR: r = x >> (b & 31); break;
          case SR_OP_MIN: r = std::min(x, y); break;
          case SR_OP_MAX: r = std::max(x, y); break;
          case SR_OP_SLT: r = x < y; break;
          case SR_OP_SLE: r = x <= y; break;
          case SR_OP_SEQ: r = x == y; break;
          case SR_OP_SNE: r = x != y; break;
          case SR_OP_S2R:
            r = im == SR_SREG_TID    ? tid
                : im == SR_SREG_BID  ? (int32_t)(first + g() % blocks)
                : im == SR_SREG_BDIM ? (int32_t)L.block_dim
                : im == SR_SREG_GDIM ? (int32_t)L.grid
                                     : 32;
            break;
          case SR_OP_BARPOPC: r = (int32_t)(g() % (L.block_dim + 1)); break;
          case SR_OP_BARAND: case SR_OP_BAROR: r = (int32_t)(g() % 2); break;
          case SR_OP_LDG: r = (int32_t)g(); break;
          case SR_OP_LDS: case SR_OP_STS: case SR_OP_ATOMS: {
            const uint32_t addr = a + (uint32_t)im;
            if (addr < shw) {
              ++accesses;
              if (addr >= reach) return printf("kernel %d pc %u: word %u, reach %u of %u\n", it, pc, addr, reach, shw), 1;
            }
            r = g() % 2 ? (int32_t)g() : (int32_t)(g() % shw);
            break;
          }
          case SR_OP_BRA: next = (uint32_t)im; break;
          case SR_OP_BRZ: if (x == 0) next = (uint32_t)im; break;
          case SR_OP_BRNZ: if (x != 0) next = (uint32_t)im; break;
          default: break;
        }
        if (op_writes_d(base) && d < 6) R[d] = r;
        pc = next;
      }
    }
  }
  printf("ok %ld %ld\n", accesses, below);
  return 0;
}
