// lb_ktrap.cuh -- the K integral of one pair on one thread (tight mode, FP64).
//
//   K_v(x) = 1/2 int_{-inf}^{inf} exp(v t - x cosh t) dt          (DLMF 10.32.9)
//
// summed by the trapezoid rule, which converges exponentially for this
// integrand: with step h the relative error is exactly
// 2 Re sum_n K_{v + 2 pi i n / h}(x) / K_v(x).  The nodes are centred at the
// integrand's maximum t0 = asinh(v/x).  With r = sqrt(v^2 + x^2),
// a = (r + v)/2, b = (r - v)/2 = x^2/(4a):
//
//   x cosh(t0 + d) = a e^d + b e^-d,     v = a - b,
//   log K = -(a + b) + v log(2a/x) + log(h/2 sum_k e^-E_k),
//   E_k = a e^(kh) + b e^(-kh) - (a + b) - v k h >= 0,
//   d/dx log K = -(1/x) sum_k (a e^(kh) + b e^(-kh)) e^-E_k / sum_k e^-E_k.
//
// Every sum has positive terms only, and no gamma function is needed.
//
// The step is h = ln2 / m.  Then a e^(kh) = (a 2^(j/m)) 2^i for k = i m + j: m
// products per pair, and after that each node's exponent is shifts and adds
// of 64-bit integers.  With everything scaled by log2(e) the exponent is a
// power of two's: its top bits are the result's shift, the next 11 a table
// index, and the rest a cubic's argument, with no reduction.  E is kept in
// Q54, the terms in Q58 and their sum (below 64) in 64 bits: about 40 integer
// instructions per node and none on the FP64 pipe, which on GB300 retires 2
// operations per SM per clock against 64 integer multiplies and 128 others.
//
// m = 3, 4, 5, 6 by a rule on (v, x) that keeps the rule's relative error
// below 1.2e-16 (kt_class); 33 to 40 nodes matter for v or x above 2, more
// towards small arguments (about 2 log2(84/x) m), where Temme's series takes
// over (kt_small, x < 2^-9).  The Gauss rules it replaces (kquad_tables.h,
// one warp per pair) evaluate 32 to 192 nodes with one logarithm and one or
// two exponentials each.
//
// The functions compile for the host too (without __CUDACC__), with the same
// results, for the CPU tests.
#pragma once

#include "lb_intmath.cuh"
#include "ktrap_tables.h"

// The per-pair functions are called, not inlined: the warps of an SM run
// several classes at a time out of one instruction cache.
#if defined(__CUDACC__)
#define LB_KT_CALL static __device__ __noinline__
#else
#define LB_KT_CALL static inline
#endif

namespace lb {

#if defined(__CUDACC__)
static __device__ __noinline__ double kt_exp(double y) { return ix_exp(y); }
LB_IX_FN double kt_log(double z) { return ix_log_call(z); }
LB_IX_FN double kt_rcp(double z) { return ix_rcp_call(z); }
LB_IX_FN double kt_rsqrt(double z) { return ix_rsqrt_call(z); }
#else
LB_IX_FN double kt_exp(double y) { return ix_exp(y); }
LB_IX_FN double kt_log(double z) { return ix_log(z); }
LB_IX_FN double kt_rcp(double z) { return ix_rcp(z); }
LB_IX_FN double kt_rsqrt(double z) { return ix_rsqrt(z); }
#endif

constexpr double kKtLn2 = 0.693147180559945309417232121458;

// High 64 bits of a 64 x 64-bit product without the carry of the lowest
// 32 x 32 bits: at most 1 below the exact value.  Three 32 x 32 -> 64-bit
// multiply-adds; needs (a >> 32) + (b >> 32) < 2^32.
LB_IX_FN uint64_t kt_mulhi(uint64_t a, uint64_t b) {
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
  uint64_t t = (uint64_t)ah * bl;
  t += (uint64_t)al * bh;
  return (uint64_t)ah * bh + (t >> 32);
}

// 2^N for N <= 0 in Q54, in Q58 (truncated); tab = lb_kt_exp2.
LB_IX_FN uint64_t kt_exp2_q58(int64_t N, const unsigned long long* tab) {
  const int k = (int)(N >> 43);                             // floor(2048 N)
  const uint64_t T = tab[k & 2047];                         // 2^((k mod 2048)/2048), Q62
  const uint64_t R = (uint64_t)N << 21;                     // the remainder r < 2^-11, Q75
  const uint32_t Rh = (uint32_t)(R >> 32), Rl = (uint32_t)R;
  // 2^r - 1 = r q, q = c1 + r (c2 + r c3): r in Q43 suffices for the inner steps
  const uint32_t b = LB_KT_C2 + (uint32_t)(((uint64_t)(LB_KT_C3 >> 11) * Rh) >> 32);   // Q33
  const uint64_t q = LB_KT_C1 + (((uint64_t)Rh * b) >> 23);                            // Q53
  const uint32_t qh = (uint32_t)(q >> 32), ql = (uint32_t)q;
  const uint64_t p = (uint64_t)Rh * qh + (((uint64_t)Rh * ql) >> 32) + (((uint64_t)Rl * qh) >> 32);   // Q64
  const uint64_t w = T + kt_mulhi(T, p);                    // Q62, in [1, 2)
  const int sh = 4 - (k >> 11);                             // to Q58
  return w >> (sh < 63 ? sh : 63);
}

// floor(log2 a) of a positive normal double, and a log2(e) 2^(62 - that).
LB_IX_FN uint64_t kt_norm(double a, int& e) {
  const uint64_t b = ix_bits(a);
  e = (int)(b >> 52) - 1023;
  return ix_umulhi(((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << 11, 0xb8aa3b295c17f0bcull);
}

// 2^(j/M), Q63, j = 1 .. M-1 (both constant after unrolling).
template <int M>
LB_IX_FN uint64_t kt_root(int j) {
  if (M == 3) return j == 1 ? LB_KT_ROOT3_1 : LB_KT_ROOT3_2;
  if (M == 4) return j == 1 ? LB_KT_ROOT4_1 : (j == 2 ? LB_KT_ROOT4_2 : LB_KT_ROOT4_3);
  if (M == 5)
    return j == 1 ? LB_KT_ROOT5_1 : (j == 2 ? LB_KT_ROOT5_2 : (j == 3 ? LB_KT_ROOT5_3 : LB_KT_ROOT5_4));
  return j == 1 ? LB_KT_ROOT6_1
       : (j == 2 ? LB_KT_ROOT6_2 : (j == 3 ? LB_KT_ROOT6_3 : (j == 4 ? LB_KT_ROOT6_4 : LB_KT_ROOT6_5)));
}

// The trapezoid sum: S in Q58 (the term at the maximum is 2^58), and for DX
// G = sum e^-E_k x cosh(t_k) log2(e) in Q54.  a2 = 2a, b2 = 2b.
// A is the factor that grows on a side (a to the right of the maximum, b to
// the left) times 2^(j/M), B the one that shrinks; A[j] >> sa is in Q54, so
// A 2^(i + j/M) is A[j] >> (sa - i).  Each side goes on by groups of M nodes
// to the first whose last term is below 2^-54 (what follows it is below
// 2^-57 of the sum).  While terms are above that, the
// growing factor stays below 2^8 through the end of its group (v <= 16.5,
// r <= 30.1), so sa - i - 1 >= 0.
template <int M, bool DX>
LB_IX_FN void kt_sum(double v, double a2, double b2, const unsigned long long* tab, uint64_t& S, uint64_t& G) {
  uint64_t A[M], B[M];
  int ea, eb;
  const uint64_t ma = kt_norm(a2, ea), mb = kt_norm(b2, eb);   // Q62 of a2, so Q63 of a, log2(e) included
  A[0] = ma >> 1;
  B[0] = mb >> 1;
#pragma unroll
  for (int j = 1; j < M; ++j) {
    A[j] = ix_umulhi(ma, kt_root<M>(j));
    B[j] = ix_umulhi(mb, kt_root<M>(j));
  }
  int sa = 8 - ea, sb = 8 - eb;                             // a's exponent is ea - 1; A is in Q(61 - (ea - 1))
  const int64_t base = (int64_t)((A[0] >> sa) + (B[0] >> (sb < 63 ? sb : 63)));
  int64_t vstep = ix_fix(v * (1.0 / M), 54);
  S = 1ull << 58;
  G = (uint64_t)base + 1;
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {                    // one copy of the code for both sides
    int64_t c = base, N = 0;
#pragma unroll 1
    for (int i = 0; i < 64 && N >= -(54ll << 54); ++i) {
      const int s0 = sa - i, s1 = s0 > 1 ? s0 - 1 : 0, sd = sb + i + 1 < 63 ? sb + i + 1 : 63;
#pragma unroll
      for (int j = 1; j <= M; ++j) {
        c += vstep;
        const int64_t t = (int64_t)((j < M ? A[j < M ? j : 0] >> s0 : A[0] >> s1) + (B[M - j] >> sd));   // x cosh t_k
        N = c - t;
        const uint64_t w = kt_exp2_q58(N, tab);
        S += w;
        if (DX) G += ix_umulhi(w << 6, (uint64_t)t + 1);    // + 1: the two shifts' mean truncation; w < 2^58
      }
      if (DX) G += M / 2;                                   // the products' mean truncation
    }
#pragma unroll
    for (int j = 0; j < M; ++j) {
      const uint64_t t = A[j];
      A[j] = B[j];
      B[j] = t;
    }
    const int t = sa;
    sa = sb;
    sb = t;
    vstep = -vstep;
  }
}

// n / d with the reciprocal's and the product's rounding corrected by the
// remainder (quotients above 2^993 as they come, infinities among them).
LB_IX_FN double kt_div(double n, double d) {
  const double r = kt_rcp(d), q = n * r;
  if ((ix_bits(q) & 0x7fffffffffffffffull) >= 0x7e00000000000000ull) return q;
  return fma(r, fma(-q, d, n), q);
}

// Temme's Gamma_1(mu) and Gamma_2(mu) in Q62 (1/Gamma(1 +- mu) = Gamma_2 -+ mu
// Gamma_1), |mu| <= 1/2 in Q62, by their Taylor series in mu^2.
LB_IX_FN void kt_gammas(int64_t mq, int64_t& g1, int64_t& g2) {
  const int64_t m2 = ix_mulhi(mq, mq) << 4;                 // mu^2, Q64
  int64_t q1 = LB_KT_G1_8, q2 = LB_KT_G2_8;
  q1 = LB_KT_G1_7 + ix_mulhi(q1, m2);
  q2 = LB_KT_G2_7 + ix_mulhi(q2, m2);
  q1 = LB_KT_G1_6 + ix_mulhi(q1, m2);
  q2 = LB_KT_G2_6 + ix_mulhi(q2, m2);
  q1 = LB_KT_G1_5 + ix_mulhi(q1, m2);
  q2 = LB_KT_G2_5 + ix_mulhi(q2, m2);
  q1 = LB_KT_G1_4 + ix_mulhi(q1, m2);
  q2 = LB_KT_G2_4 + ix_mulhi(q2, m2);
  q1 = LB_KT_G1_3 + ix_mulhi(q1, m2);
  q2 = LB_KT_G2_3 + ix_mulhi(q2, m2);
  q1 = LB_KT_G1_2 + ix_mulhi(q1, m2);
  q2 = LB_KT_G2_2 + ix_mulhi(q2, m2);
  q1 = LB_KT_G1_1 + ix_mulhi(q1, m2);
  q2 = LB_KT_G2_1 + ix_mulhi(q2, m2);
  q1 = LB_KT_G1_0 + ix_mulhi(q1, m2);
  q2 = LB_KT_G2_0 + ix_mulhi(q2, m2);
  g1 = q1;
  g2 = q2;
}

// Small arguments, x < 2^-9, v <= 16.5: Temme's series for K_mu and
// K_(mu+1), v = n + mu, |mu| <= 1/2 (J. Comput. Phys. 19, 1975; y = x^2/4 <
// 2^-20, so two terms past the leading one), then n steps of
// K_(u+1) = K_(u-1) + (2u/x) K_u, on (x/2)^(u - mu) K_u, which neither
// overflows nor divides.  Gamma_1 and Gamma_2 are summed in integers.
template <bool DX>
LB_IX_FN double kt_small(double v, double x) {
  const int n = (int)(v + 0.5);
  double mu = v - (double)n;
  const double L = kKtLn2 - kt_log(x);                      // log(2/x) >= 6.9
  int64_t q1, q2;
  kt_gammas(ix_fix(mu, 62), q1, q2);
  const double G1 = (double)q1 * 0x1p-62, G2 = (double)q2 * 0x1p-62;
  const double mg = mu * G1;
  const double gp = kt_rcp(G2 - mg), gm = kt_rcp(G2 + mg);   // Gamma(1 + mu), Gamma(1 - mu)
  const double s = mu * L;
  const double ep = kt_exp(s), em = kt_rcp(ep);
  double shc;                                               // sinh(s) / s
  if (fabs(s) < 0.5) {
    const double z = s * s;
    shc = 1.0 / 1307674368000.0;
    shc = fma(shc, z, 1.0 / 6227020800.0);
    shc = fma(shc, z, 1.0 / 39916800.0);
    shc = fma(shc, z, 1.0 / 362880.0);
    shc = fma(shc, z, 1.0 / 5040.0);
    shc = fma(shc, z, 1.0 / 120.0);
    shc = fma(shc, z, 1.0 / 6.0);
    shc = fma(shc, z, 1.0);
  } else {
    shc = (ep - em) * (0.5 * kt_rcp(fabs(s)));
    shc = s < 0.0 ? -shc : shc;
  }
  double f = gp * gm * fma(0.5 * (ep + em), G1, shc * L * G2);
  double p = 0.5 * ep * gp, q = 0.5 * em * gm;
  if (DX && n == 0) {                                       // the derivative takes K_(1-mu) there: the roles swapped
    const double t = p;
    p = q;
    q = t;
    mu = -mu;
  }
  const double y = 0.25 * x * x;
  const double w = mu * mu;
  const double r1 = kt_rcp(1.0 - w), r2 = kt_rcp(4.0 - w);
  double s0 = f, s1 = p;
  f = (f + p + q) * r1;                                     // k = 1: c = y
  p *= (1.0 + mu) * r1;
  q *= (1.0 - mu) * r1;
  s0 = fma(y, f, s0);
  s1 = fma(y, p - f, s1);
  f = (fma(2.0, f, p) + q) * r2;                            // k = 2: c = y^2/2
  p *= (2.0 + mu) * r2;
  const double c2 = 0.5 * y * y;
  s0 = fma(c2, f, s0);
  s1 = fma(c2, fma(-2.0, f, p), s1);
  // s0 = K_mu, s1 = (x/2) K_(mu+1); d/dx log K_v = -v/x - K_(v-1)/K_v
  if (n == 0) {
    if (DX) return -kt_div(fma(2.0 * s1, kt_rcp(s0), v), x);
    return kt_log(s0);
  }
  double u = mu + 1.0;
#pragma unroll 1
  for (int k = 1; k < n; ++k) {
    const double t = fma(u, s1, y * s0);
    s0 = s1;
    s1 = t;
    u += 1.0;
  }
  if (DX) return -kt_div(fma(2.0 * y * s0, kt_rcp(s1), v), x);
  return fma((double)n, L, kt_log(s1));
}

// Any (v, x) with finite r (pairs outside the other classes' ranges, which
// only a forced evaluation reaches): the same sum in FP64 with the library
// functions, h = min(ln2 / 6, 0.45 / sqrt(r)) -- the integrand's width is
// 1/sqrt(r) -- where the rule's error is below 1e-20.
template <bool DX>
LB_KT_CALL double kt_any(double v, double x) {
  const double r = hypot(v, x), a2 = r + v, b2 = x * (x / a2);
  const double h = fmin(0.11552453009332422, 0.45 / sqrt(r));
  double S = 1.0, G = r;
  for (int side = 0; side < 2; ++side)
    for (int k = 1; k < 8192; ++k) {
      const double d = side ? -h * k : h * k;
      const double ed = expm1(d), em = expm1(-d);
      const double E = 0.5 * (a2 * (ed - d) + b2 * (em + d));
      const double w = exp(-E);
      S += w;
      if (DX) G += w * 0.5 * fma(a2, ed + 1.0, b2 * (em + 1.0));
      if (!(E < 45.0)) break;
    }
  if (DX) return -(G / S) / x;
  return fma(v, log(a2 / x), -0.5 * (a2 + b2)) + log(0.5 * h * S);
}

// Class of a pair, costliest first: 0 any other pair (kt_any), 1 the
// trapezoid rule with m = 3, 2 the small-argument series, 3, 4, 5 the
// trapezoid rule with m = 6, 5, 4.  The edges of m keep
// 2 |K_(v + 2 pi i m / ln2)(x)| / K_v(x) below 1.2e-16 (measured over the
// region in 30 digits); the x-derivative's sum is K_(v+1)'s and takes its
// edges.  In single precision: a pair next to an edge may land on either
// side of it, both sides being accurate there.
LB_IX_FN int kt_class(double v, double x, bool dx) {
  const float vf = (float)v, xf = (float)x;
  if (!(vf <= 16.5f)) return 0;
  if (xf < 0x1p-9f) return 2;
  const float ve = dx ? vf + 1.0f : vf, v2 = ve * ve;
  if (xf <= fmaf(-1.5f, v2, 4.5f)) return 1;
  if (xf <= fmaf(-0.28f, v2, 17.8f)) return 5;
  if (xf <= fmaf(-0.09f, v2, 31.0f)) return 4;
  return fmaf(xf, xf, vf * vf) <= 901.0f ? 3 : 0;
}

// Band 0 .. 7 of a pair within its class, by an estimate of its work, so
// that pairs sorted by it make warps whose lanes finish together (it changes
// no result): the doublings of each side until a e^d (right) or b e^-d or
// v d (left) reaches the cutoff, or the recurrence's steps in class 2.
LB_IX_FN int kt_band(double v, double x, int cls) {
  const float vf = (float)v, xf = (float)x;
  if (cls == 2) return (int)(0.46f * vf);
  if (cls == 0) return 0;
  const float a2 = vf + sqrtf(fmaf(vf, vf, xf * xf));       // 2a; 2b = x^2/a2
  const float right = log2f(2.0f + 80.0f / a2);
  const float left = fminf(log2f(2.0f + 80.0f * a2 / (xf * xf)), (41.0f + 0.5f * a2) / (0.7f * vf));
  const float w = 3.2f * log2f((right + left) * (cls == 1 ? 0.125f : 0.25f));
  return w < 0.0f ? 0 : (w > 7.0f ? 7 : (int)w);
}

// log K (DX = false) or d/dx log K of one pair of class cls, v >= 0, x > 0.
template <bool DX>
LB_IX_FN double kt_eval(double v, double x, int cls, const unsigned long long* tab) {
  if (cls == 2) return kt_small<DX>(v, x);
  if (cls == 0) return kt_any<DX>(v, x);
  const double r2 = fma(v, v, x * x);
  const double a2 = fma(r2, kt_rsqrt(r2), v);               // r + v = 2a
  const double b2 = x * x * kt_rcp(a2);                     // r - v = 2b
  uint64_t S, G;
  switch (cls) {
    case 1: kt_sum<3, DX>(v, a2, b2, tab, S, G); break;
    case 5: kt_sum<4, DX>(v, a2, b2, tab, S, G); break;
    case 4: kt_sum<5, DX>(v, a2, b2, tab, S, G); break;
    default: kt_sum<6, DX>(v, a2, b2, tab, S, G); break;
  }
  // Q54 over Q58, base 2 to e: 16 ln2 in Q60
  if (DX) return -kt_div((double)ix_umulhi(G, 0xb17217f7d1cf79acull) * 16.0, (double)S * x);
  // h/2 = ln2 / (2m)
  const double hh = cls == 1 ? kKtLn2 / 6.0 : (cls == 5 ? kKtLn2 / 8.0 : (cls == 4 ? kKtLn2 / 10.0 : kKtLn2 / 12.0));
  return fma(v, kt_log(a2 * kt_rcp(x)), fma(-0.5, a2 + b2, kt_log((double)S * (0x1p-58 * hh))));
}

}  // namespace lb
