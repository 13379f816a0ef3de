// Host check of shared_reach_of: over the launches of a program - other parameters, block sizes and
// grids in any order - it gives what the analysis of each launch by itself gives (kernels without
// loops: there one analysis does not depend on the order in which intervals arrive), and it analyses a
// kernel whose addresses do not follow from the parameters once per shape.  Prints "ok <launches>
// <analyses>" or the first difference.
#include <cstdio>
#include <random>
#include <vector>

#include "host_prep.h"

using namespace sr;
using namespace sr::host;

int main() {
  const uint32_t alu[17] = {SR_OP_MOV, SR_OP_ADD, SR_OP_SUB, SR_OP_MUL, SR_OP_DIV, SR_OP_REM, SR_OP_AND, SR_OP_OR, SR_OP_XOR,
                            SR_OP_SHL, SR_OP_SHR, SR_OP_MIN, SR_OP_MAX, SR_OP_SLT, SR_OP_SLE, SR_OP_SEQ, SR_OP_SNE};
  std::mt19937 g(11);
  RangeScratch memo, fresh;
  long launches = 0;
  for (int it = 0; it < 4000; ++it) {
    const uint32_t n = 4 + g() % 30;
    std::vector<sr_instr> code(n);
    auto reg = [&]() { return g() % 16 == 0 ? (uint32_t)SR_RZ : (uint32_t)(g() % 6); };
    for (uint32_t i = 0; i < n; ++i) {
      const uint32_t d = reg(), a = reg(), b = reg(), what = g() % 14;
      int32_t im = (int32_t)(g() % 80) - 16;
      uint32_t op = alu[g() % 17] | (g() % 2 ? SR_BIMM : 0u);
      if (what < 3) op = SR_OP_AND | SR_BIMM;
      else if (what < 5) op = g() % 2 ? SR_OP_STS : SR_OP_LDS;
      else if (what == 5) { op = SR_OP_S2R; im = (int32_t)(g() % 5); }
      else if (what == 6) { op = g() % 2 ? SR_OP_BRZ : SR_OP_BRNZ; im = (int32_t)(i + 1 + g() % (n - i)); }
      code[i] = {op | d << 8 | a << 16 | b << 24, im};
    }
    memo.seen.clear();
    for (int l = 0; l < 12; ++l) {
      sr_launch L{};
      L.grid = 1 + g() % 2;
      L.block_dim = 32u << g() % 2;
      L.shmem_words = 1000 + 1000 * (g() % 2);
      L.nparams = g() % 3;
      for (uint32_t q = 0; q < L.nparams; ++q) L.params[q] = (int32_t)(g() % 200) - 50;
      const uint32_t got = shared_reach_of(code.data(), n, 0, L, memo), want = shared_reach(code.data(), n, 0, L, fresh);
      if (got != want) return printf("kernel %d launch %d: %u, by itself %u\n", it, l, got, want), 1;
      ++launches;
    }
  }
  // a long kernel, two hundred launches that differ in a parameter of theirs: analysed once
  std::vector<sr_instr> code(3000, sr_instr{SR_OP_ADD | SR_BIMM | 5u << 8 | 5u << 16, 1});
  code[0] = {SR_OP_S2R | 2u << 8, SR_SREG_TID};
  code[2998] = {SR_OP_STS | 2u << 16 | 0u << 24, 0};
  code[2999] = {SR_OP_EXIT, 0};
  memo.seen.clear();
  memo.analyses = 0;
  for (int l = 0; l < 200; ++l) {
    sr_launch L{};
    L.grid = 1; L.block_dim = 64; L.shmem_words = 100; L.nparams = 1; L.params[0] = l;
    if (shared_reach_of(code.data(), 3000, 0, L, memo) != 64) return printf("long kernel, launch %d\n", l), 1;
  }
  if (memo.analyses != 1) return printf("%llu analyses of one kernel\n", (unsigned long long)memo.analyses), 1;
  printf("ok %ld %llu\n", launches, (unsigned long long)memo.analyses);
  return 0;
}
