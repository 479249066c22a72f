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
// logarithms within 2^-53, against a result of the size of r >= 16.  Bound by
// issue and the integer multiplies.  log K over mixed orders, 22M pairs: 1.89
// -> 1.56 ms with these sums in place of FP64 with double-float tails, 1.54
// with the outer sums biased to stay positive; log K and its derivative, 4M:
// 880 -> 742 us with the derivative's too.  Loops unrolled by two or three
// were slower (instruction fetch).
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

// The sums' variables from v/r <= 1 and 1/r: g = p/2, y = p^2/2, h = 8/r
// (below 1/2), all in Q64.  The outer sums run over +-h and are kept with
// kUniBias added, so that they stay positive and take the short unsigned
// product; hb is the bias's product with h.
struct UniVars {
  uint64_t g, y, h, hb;
};
constexpr uint64_t kUniBias = 1ull << 57;
LB_IX_FN UniVars uni_vars(double vr, double q) {
  UniVars u;
  const uint64_t t = (uint64_t)ix_fix(vr, 62);
  u.g = kt_mulhi(t, t) << 3;
  u.y = kt_mulhi(u.g >> 1, u.g >> 1) << 3;
  u.h = (uint64_t)ix_fix(q, 67);
  u.hb = u.h >> 7;                                          // 2^57 h / 2^64
  return u;
}
// kUniBias +- h (acc - kUniBias), c0 = kUniBias -+ hb.
LB_IX_FN uint64_t uni_step(int kind, uint64_t acc, uint64_t h, uint64_t c0) {
  const uint64_t m = kt_mulhi(acc, h);
  return kind ? c0 - m : c0 + m;
}

// log I (kind 0) or log K from the sum S (Q62, below 2), r and q = 1/r.  r and
// v log(x/(v + r)) first, which nearly cancel where the result is small: the
// rest is then added to what is left, not rounded to the size of r before.
LB_IX_FN double uni_log(int kind, double v, double x, double r, double q, uint64_t S) {
  // S^2 / r: Q62 x Q62, then the 53 bits of 1/r
  const uint64_t bq = ix_bits(q);
  const uint64_t W = kt_mulhi(kt_mulhi(S, S) << 2, ((bq & 0x000fffffffffffffull) | 0x0010000000000000ull) << 10);   // Q60
  const long long lw = kt_logq(ix_pack(W, 1021 - (int)(bq >> 52)));
  const double a = (double)(kt_logq(x) - kt_logq(v + r)), w = v * 0x1p-53;
  const double e = fma(w, a, r);
  if (kind == 0) return fma(0x1p-54, (double)(lw - kHalfLog2PiQ53x2), e);
  return fma(0x1p-54, (double)(lw + kLogHalfPiQ53), -e);
}

// log I (kind 0) or log K of one pair with s = v^2 + x^2, uni_ok; K: the
// pair's terms, Kmax: the warp's largest.
LB_IX_FN double u_fx(int kind, double v, double x, double s, int K, int Kmax) {
  const double q = kt_rsqrt(s), r = s * q;                  // 1/r, r
  const UniVars u = uni_vars(v * q, q);
  const uint64_t c0 = kind ? kUniBias + u.hb : kUniBias - u.hb;
  uint64_t acc = kUniBias;
#pragma unroll 1
  for (int k = Kmax; k >= 1; --k) {
    const int b = lb_uni_off[k];
    int i = lb_uni_off[k + 1] - 1;
    uint64_t e = lb_uni[i][0], o = lb_uni[i][1];
#pragma unroll 1
    for (--i; i >= b; --i) {
      e = lb_uni[i][0] + kt_mulhi(e, u.y);
      o = lb_uni[i][1] + kt_mulhi(o, u.y);
    }
    acc = uni_step(kind, acc, u.h, c0) + e - kt_mulhi(o, u.g);
    if (k > K) acc = kUniBias;
  }
  const uint64_t S = uni_step(kind, acc, u.h, c0) + (1ull << 56) - kUniBias;   // Q56
  return uni_log(kind, v, x, r, q, S << 6);
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
  const UniVars u = uni_vars(v * q, q);
  const uint64_t c0 = kind ? kUniBias + u.hb : kUniBias - u.hb;
  uint64_t acc = kUniBias, dcc = kUniBias;
#pragma unroll 1
  for (int k = Kmax; k >= 1; --k) {
    const int b = lb_uni_off[k];
    int i = lb_uni_off[k + 1] - 1;
    uint64_t e = lb_uni[i][0], o = lb_uni[i][1], de = lb_uniq[i][0], dd = lb_uniq[i][1];
#pragma unroll 1
    for (--i; i >= b; --i) {
      e = lb_uni[i][0] + kt_mulhi(e, u.y);
      o = lb_uni[i][1] + kt_mulhi(o, u.y);
      de = lb_uniq[i][0] + kt_mulhi(de, u.y);
      dd = lb_uniq[i][1] + kt_mulhi(dd, u.y);
    }
    acc = uni_step(kind, acc, u.h, c0) + e - kt_mulhi(o, u.g);
    dcc = uni_step(kind, dcc, u.h, c0) + de - kt_mulhi(dd, u.g);
    if (k > K) acc = dcc = kUniBias;
  }
  const double S = (double)(int64_t)(uni_step(kind, acc, u.h, c0) + (1ull << 56) - kUniBias);   // Q56
  const double SQ = (double)(int64_t)(uni_step(kind, dcc, u.h, c0) - kUniBias) * 64.0;           // Q50 to Q56
  const double corr = (x * q) * q * fma(SQ, kt_rcp(S), 0.5);
  const double lead = r * kt_rcp(x);
  return kind ? -lead - corr : lead - corr;
}

}  // namespace lb
