// lb_uniform.cuh -- the uniform large-order expansion in fixed point (values).
//
// The same sums as U_K (paper Eqs. "log Iv u k", "log Kv u k"), in the
// variables of the pair rather than of the order: with r = sqrt(v^2 + x^2),
// p = (v/r)^2 and u_k(t) = t^k P_k(t^2), t = v/r,
//   log I = -log(2 pi r)/2 + r + v (log x - log(v + r)) + log S,  S = 1 + sum_k P_k(p) / r^k,
//   log K =  log(pi/(2r))/2 - r - v (log x - log(v + r)) + log S,  S = 1 + sum_k P_k(p) / (-r)^k.
// One 1/sqrt gives r, 1/r and p; no reciprocal of v and no division.
//
// On GB300 an FP64 operation costs the time of 64 issue slots of a thread's
// lane, a double-float step 15, and a 64-bit fixed-point multiply-add about 6:
// the polynomials, S and S^2/r are integers (Q56, variables Q64 halved so that
// they stay below 2^63), and the three logarithms come in Q53 straight from
// ix_log_q53; nine FP64 operations are left.  S is within 2^-54 and the
// logarithms within 2^-53, against a result of the size of r >= 16.
//
// K is the pair's own: the cap of its region (4, 6, 9, 13 by the order), or
// less where r is large enough (uni_terms).  Lanes with a smaller K than the
// warp's hold a zero sum until their first term, so a pair's result does not
// depend on its warp.
//
// The functions compile for the host too (without __CUDACC__).
#pragma once

#include "lb_intmath.cuh"
#include "lb_ktrap.cuh"
#include "uniform_tables.h"

namespace lb {

constexpr long long kHalfLog2PiQ53x2 = 16554124942867817ll;   // log(2 pi), Q53
constexpr long long kLogHalfPiQ53 = 4067495406537099ll;       // log(pi/2), Q53

#if defined(__CUDACC__)
static __device__ __noinline__ long long kt_logq(double z) { return ix_log_q53(z); }
#else
LB_IX_FN long long kt_logq(double z) { return ix_log_q53(z); }
#endif

// Terms that a pair with r^2 = s needs, at most cap: the smallest K with
// max|P_(K+1)| / r^(K+1) <= 3e-17 r (the result is of the size of r or
// larger), by half octaves of s from 768, 13 below, 4 from 1.5 2^17.
// f: s in single precision.
LB_IX_FN int uni_terms(float f, int cap) {
  const int i = (int)(ix_fbits(f) >> 22) - (2 * (127 + 9) + 1);
  const int K = i < 0 ? 13 : (i > 15 ? 4 : (int)((0x555566677889abcdull >> (4 * i)) & 15u));
  return K < cap ? K : cap;
}

// Whether u_fx applies: r in [16.04, 1e150], x normal.
LB_IX_FN bool uni_ok(double s, double x) {
  const uint32_t hs = (uint32_t)(ix_bits(s) >> 32), hx = (uint32_t)(ix_bits(x) >> 32);
  return hs >= 0x40701000u && hs < 0x7e37e43cu && hx >= 0x00100000u;
}

// log I (kind 0) or log K of one pair with s = v^2 + x^2, uni_ok; K: the
// pair's terms, Kmax: the warp's largest.
LB_IX_FN double u_fx(int kind, double v, double x, double s, int K, int Kmax) {
  const double q = kt_rsqrt(s), r = s * q;                  // 1/r, r
  const uint64_t t = (uint64_t)ix_fix(v * q, 63);           // v/r <= 1
  const uint64_t g = ix_umulhi(t, t) << 1;                  // p/2 in Q64
  const uint64_t y = ix_umulhi(g, g) << 1;                  // p^2/2 in Q64
  const int64_t h = kind ? -ix_fix(q, 67) : ix_fix(q, 67);  // +-8/r in Q64, below 1/2
  int64_t acc = 0;
#pragma unroll 1
  for (int k = Kmax; k >= 1; --k) {
    const int b = lb_uni_off[k];
    int i = lb_uni_off[k + 1] - 1;
    uint64_t e = lb_uni[i][0], o = lb_uni[i][1];
#pragma unroll 1
    for (--i; i >= b; --i) {
      e = lb_uni[i][0] + kt_mulhi(e, y);
      o = lb_uni[i][1] + kt_mulhi(o, y);
    }
    acc = ix_mulhi(acc, h) + (int64_t)(e - kt_mulhi(o, g));
    if (k > K) acc = 0;
  }
  const uint64_t S = (uint64_t)((1ll << 56) + ix_mulhi(acc, h));      // Q56
  // S^2 / r: Q63 x Q63, then the 53 bits of 1/r
  const uint64_t bq = ix_bits(q);
  const uint64_t W = ix_umulhi(ix_umulhi(S << 7, S << 7), ((bq & 0x000fffffffffffffull) | 0x0010000000000000ull) << 11);   // Q61
  const long long lw = kt_logq(ix_pack(W, 1022 - (int)(bq >> 52)));
  const double a = (double)(kt_logq(x) - kt_logq(v + r)), w = v * 0x1p-53;
  if (kind == 0) return fma(w, a, fma(0x1p-54, (double)(lw - kHalfLog2PiQ53x2), r));
  return -fma(w, a, fma(-0x1p-54, (double)(lw + kLogHalfPiQ53), r));
}

// Terms for the x-derivative, whose sum's term k is k times the value's: the
// value's rule at r/1.31 (1.31 = 5^(1/6), the most that (K + 1)^(1/(K + 2)) is).
LB_IX_FN int uni_terms_dx(float f, int cap) { return uni_terms(f * 0.58f, cap); }

// d/dx log I or log K of one pair, arguments as u_fx (K: uni_terms_dx).  r
// alone depends on x:
//   d/dx log f = +-r/x - (x/r^2) (1/2 + SQ/S),  SQ = sum_k (+-1/r)^k Q_k(p),
// Q_k = k P_k + 2 p P_k'.  SQ is below 0.3/r of a factor that is below 1/r of
// the result: its 2^-50 and S's 2^-56 are far below the result's last place.
LB_IX_FN double u_dx_fx(int kind, double v, double x, double s, int K, int Kmax) {
  const double q = kt_rsqrt(s), r = s * q;
  const uint64_t t = (uint64_t)ix_fix(v * q, 63);
  const uint64_t g = ix_umulhi(t, t) << 1;
  const uint64_t y = ix_umulhi(g, g) << 1;
  const int64_t h = kind ? -ix_fix(q, 67) : ix_fix(q, 67);
  int64_t acc = 0, dcc = 0;
#pragma unroll 1
  for (int k = Kmax; k >= 1; --k) {
    const int b = lb_uni_off[k];
    int i = lb_uni_off[k + 1] - 1;
    uint64_t e = lb_uni[i][0], o = lb_uni[i][1], de = lb_uniq[i][0], dd = lb_uniq[i][1];
#pragma unroll 1
    for (--i; i >= b; --i) {
      e = lb_uni[i][0] + kt_mulhi(e, y);
      o = lb_uni[i][1] + kt_mulhi(o, y);
      de = lb_uniq[i][0] + kt_mulhi(de, y);
      dd = lb_uniq[i][1] + kt_mulhi(dd, y);
    }
    acc = ix_mulhi(acc, h) + (int64_t)(e - kt_mulhi(o, g));
    dcc = ix_mulhi(dcc, h) + (int64_t)(de - kt_mulhi(dd, g));
    if (k > K) acc = dcc = 0;
  }
  const double S = (double)((1ll << 56) + ix_mulhi(acc, h));          // Q56
  const double SQ = (double)ix_mulhi(dcc, h) * 64.0;                  // Q50 to Q56
  const double corr = (x * q) * q * fma(SQ, kt_rcp(S), 0.5);
  const double lead = r * kt_rcp(x);
  return kind ? -lead - corr : lead - corr;
}

}  // namespace lb
