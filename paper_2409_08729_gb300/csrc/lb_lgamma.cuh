// lb_lgamma.cuh -- lgamma(v + 1) for the power series of log I, in integers.
//
// The library's lgamma costs 28 FP64 operations on equal arguments and takes
// several of its branches in a warp of mixed orders; on GB300 one FP64
// operation costs the time of 64 issue slots.  The series is taken for
// v <= 16 only, so here t = v + 1 in [1, 18) selects one of 33 pieces (eight
// per octave) and a polynomial of degree 12 in Q57 gives the value: no
// branch, no FP64 operation but the last conversion, error below 2e-17
// absolute before its rounding (Horner's rule in s/8: each step's truncation
// of 2^-57 counts an eighth in the next).
// log I over the whole domain, per-pair orders, 8M pairs: 1160 -> 575 us (FP64
// pipe 80 % busy before, issue 35 %); mixed sweep orders 630 -> 558.
//
// The function compiles for the host too (without __CUDACC__).
#pragma once

#include "lb_intmath.cuh"
#include "lgamma_table.h"

namespace lb {

LB_IX_FN bool lg_ok(double v) { return (uint32_t)(ix_bits(v) >> 32) < 0x40310000u; }   // 0 <= v < 17

LB_IX_FN double lg_lgamma1p(double v) {
  const uint64_t T = (uint64_t)ix_fix(v, 58) + (1ull << 58);    // t, Q58
  const int lz = ix_clz(T);
  const uint64_t r = T << (lz + 1);                             // below the leading bit
  const int row = 8 * (5 - lz) + (int)(r >> 61);
  const int64_t s = (int64_t)((r << 3) ^ 0x8000000000000000ull);   // [-1, 1), Q63
  int64_t a = (int64_t)LB_IX_LOAD(&lb_lg[row][0]);
#pragma unroll 4
  for (int k = 1; k <= LB_LG_DEG; ++k) a = (int64_t)LB_IX_LOAD(&lb_lg[row][k]) + (ix_mulhi(a, s) >> 2);
  return (double)a * 0x1p-57;
}

}  // namespace lb
