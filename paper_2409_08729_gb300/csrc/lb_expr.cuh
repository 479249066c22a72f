// lb_expr.cuh -- per-pair expressions of the log-Bessel algorithm (device code).
//
// Each function evaluates one of the paper's expressions for one (v, x) pair
// in double precision:
//   mu_K  : large-argument expansion (paper Sec. 3.1 Eq. "log Iv mu k",
//           Sec. 3.2 Eq. "log Kv mu k")
//   U_K   : uniform large-order expansion (Eqs. "log Iv u k", "log Kv u k")
//   series: power series of I_v summed in log scale (Eqs. "Iv infinite series",
//           "ak recurrence", "log Iv")
// U_K values and derivatives in tight mode run in fixed point (lb_uniform.cuh).
// The K integral (Eq. "log Kv integral") is in lb_ktrap.cuh (tight mode, one
// pair per thread) and lb_kint.cuh (the paper's Simpson rule, warp-cooperative).
#pragma once

#include <math.h>
#include <stdint.h>

template <typename T> __host__ __device__ __forceinline__ T lb_fma(T a, T b, T c);
template <> __host__ __device__ __forceinline__ double lb_fma<double>(double a, double b, double c) { return fma(a, b, c); }
template <> __host__ __device__ __forceinline__ float lb_fma<float>(float a, float b, float c) { return fmaf(a, b, c); }

#include "lb_df.cuh"
#include "debye_uk.h"
#include "lb_fastmath.cuh"
#include "lb_intmath.cuh"
#include "lb_uniform.cuh"
#include "lb_lgamma.cuh"
#include "lb_order.cuh"

namespace lb {

constexpr double kPi = 3.141592653589793238462643383279502884;
constexpr double kTwoPi = 6.283185307179586476925286766559005768;
constexpr double kHalfLogPi = 0.5723649429247000870717136756012478;   // log(pi)/2
constexpr double kHalfLog2Pi = 0.9189385332046727417803297364056177;  // log(2 pi)/2
constexpr double kHalfLogHalfPi = 0.2257913526447274323630976149;     // log(pi/2)/2

enum Kind { KIND_I = 0, KIND_K = 1 };
enum Region { R_MU20 = 0, R_U13 = 1, R_FALLBACK = 2, R_SPECIAL = 3, R_MU3 = 4, R_U4 = 5, R_U6 = 6, R_U9 = 7 };
enum Mode { MODE_TIGHT = 0, MODE_PAPER_GPU = 1, MODE_PAPER_CPU = 2 };

// ---------------------------------------------------------------------------
// Domain edges (shared convention of the library): returns true and sets *r
// when (v, x) is an edge case; K callers pass |v|.
// ---------------------------------------------------------------------------
// The tests use the IEEE bit patterns (integer instructions): on GB300 a
// double-precision compare costs as much FP64-pipe time as an FMA.
__device__ __forceinline__ bool bits_nan(long long b) { return (b & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL; }
__device__ __forceinline__ bool bits_inf(long long b) { return (b & 0x7fffffffffffffffLL) == 0x7ff0000000000000LL; }
__device__ __forceinline__ bool bits_zero(long long b) { return (b & 0x7fffffffffffffffLL) == 0; }
__device__ __forceinline__ bool bits_neg(long long b) { return b < 0 && !bits_zero(b); }

template <int KIND>
__device__ __forceinline__ bool special_value(double v, double x, double* r) {
  const long long bv = __double_as_longlong(v), bx = __double_as_longlong(x);
  if ((bv & 0x7ff0000000000000LL) != 0x7ff0000000000000LL && (bx & 0x7ff0000000000000LL) != 0x7ff0000000000000LL &&
      !bits_neg(bx) && !bits_zero(bx) && (KIND == KIND_K || !bits_neg(bv)))
    return false;                                   // the common case: finite, x > 0, v >= 0 for I
  if (KIND == KIND_I) {
    if (bits_nan(bv) || bits_nan(bx) || bits_neg(bv) || bits_neg(bx) || (bits_inf(bv) && bits_inf(bx))) { *r = __longlong_as_double(0x7ff8000000000000LL); return true; }
    if (bits_inf(bx)) { *r = INFINITY; return true; }
    if (bits_inf(bv)) { *r = -INFINITY; return true; }
    if (bits_zero(bx)) { *r = bits_zero(bv) ? 0.0 : -INFINITY; return true; }
  } else {
    if (bits_nan(bv) || bits_nan(bx) || bits_neg(bx) || (bits_inf(bv) && bits_inf(bx))) { *r = __longlong_as_double(0x7ff8000000000000LL); return true; }
    if (bits_inf(bx)) { *r = -INFINITY; return true; }
    if (bits_zero(bx) || bits_inf(bv)) { *r = INFINITY; return true; }
  }
  return false;
}

// Domain edges of the x-derivatives: d/dx log I_v at x = 0 is 0 for v = 0
// (I_0 = 1 + x^2/4 + ...) and +inf otherwise (I_v ~ (x/2)^v / Gamma(v+1));
// d/dx log K_v at x = 0 is -inf; at x = +inf the derivatives tend to +1 (I)
// and -1 (K); an infinite order gives NaN.
template <int KIND>
__device__ __forceinline__ bool special_dx(double v, double x, double* r) {
  const double qnan = __longlong_as_double(0x7ff8000000000000LL);
  if (isnan(v) || isnan(x) || x < 0.0 || isinf(v)) { *r = qnan; return true; }
  if (KIND == KIND_I && v < 0.0) { *r = qnan; return true; }
  if (isinf(x)) { *r = (KIND == KIND_I) ? 1.0 : -1.0; return true; }
  if (x == 0.0) { *r = (KIND == KIND_I) ? (v == 0.0 ? 0.0 : INFINITY) : -INFINITY; return true; }
  return false;
}

// ---------------------------------------------------------------------------
// Region predicates (paper Table "input ranges", Algorithm 1).
// ---------------------------------------------------------------------------
// Paper thresholds as printed.  Comparisons are strict, so a pair exactly on
// a threshold falls through to the next branch.
__device__ __forceinline__ bool paper_mu3(double v, double x) {
  return (x > 1400.0 && v < 3.05) || ((0.6229 * log(x) - 3.2318 > log(v)) && v > 3.1);
}
__device__ __forceinline__ bool paper_mu20(double v, double x) {
  return (x > 30.0 && v < 15.3919) || ((0.5113 * log(x) + 0.7939 > log(v)) && x > 59.6925);
}
__device__ __forceinline__ bool paper_u4(double v, double x) { return (x > 274.2377 && v > 0.3) || v > 163.6993; }
__device__ __forceinline__ bool paper_u6(double v, double x) { return (x > 84.4153 && v > 0.46) || v > 56.9971; }
__device__ __forceinline__ bool paper_u9(double v, double x) { return (x > 35.9074 && v > 0.6) || v > 20.1534; }
__device__ __forceinline__ bool paper_u13(double v, double x) { return (x > 19.6931 && v > 0.7) || v > 12.6964; }

// Tight thresholds: the same two expressions, with the regions shrunk until
// the truncation error of mu_20 and U_13 (measured against an
// extended-precision reference on both sides of every boundary) is below
// 3e-16 of the error scale.  The curved mu_20 boundary
// 0.5113 log x + 0.7939 > log v is replaced by v^2 < 3.24 x, which follows
// the actual validity limit of the large-argument series (its terms grow like
// (v^2 / 2x)^k / k!) and needs no logarithm.
// Threshold compares of non-negative doubles on their bit patterns (same
// order as the values; integer instructions).
#define LB_GT(a, c) (__double_as_longlong(a) > __double_as_longlong(c))
#define LB_LT(a, c) (__double_as_longlong(a) < __double_as_longlong(c))
#define LB_GE(a, c) (!LB_LT(a, c))
#define LB_LE(a, c) (!LB_GT(a, c))
// A double cut (truncated) to single precision from its bit fields (signed
// 0 below 2^-126, signed inf from 2^128 up; NaN not expected): integer
// instructions, no FP64 conversion instruction.  For the single-precision
// estimates (edges, term counts) of the FP64 expressions.
__device__ __forceinline__ float f32_cut(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const unsigned sgn = (unsigned)(b >> 32) & 0x80000000u;
  const int e = (int)((b >> 52) & 0x7ff) - 1023;
  if (e < -126) return __uint_as_float(sgn);
  if (e > 127) return __uint_as_float(sgn | 0x7f800000u);
  return __uint_as_float(sgn | ((unsigned)(e + 127) << 23) | (unsigned)((b >> 29) & 0x7fffffu));
}
// The curved edge v^2 < 3.24 x in single precision: it moves the edge by at
// most a few 1e-7 relative, where the truncation error of mu_20 changes by
// as little, and spares every pair three FP64 instructions.
__device__ __forceinline__ bool tight_mu20(double v, double x) {
  if (LB_GT(x, 30.0) && LB_LT(v, 13.6)) return true;
  if (!LB_GT(x, 59.6925)) return false;
  const float vf = f32_cut(v);
  return vf * vf < 3.24f * f32_cut(x);
}
__device__ __forceinline__ bool tight_u13(double v, double x) { return (LB_GT(x, 25.0) && LB_GT(v, 0.7)) || LB_GT(v, 16.0); }

// Values (not the x-derivatives) take mu_20 and U_13 further into the
// fallback region than the shared thresholds: the truncation error of both
// expansions, measured the same way for each function (exact arithmetic of
// the truncated sums against the oracle, 1500 random points per added
// range, half of them at its edges), stays at or below 3.1e-16 of the error
// scale in
//   log K:  mu_20  x > 18.5, v < 9.5;  x > 20, v < 12.5;  x > 22, v < 13.6
//           U_13   x > 19, v > 10;     x > 14, v > 14
//   log I:  mu_20  x > 19, v < 4.5;    x > 21, v < 7.5;   x > 23, v < 9.5
//           U_13   x > 19.5, v > 10;   x > 17.5, v > 12;  x > 14.5, v > 14
// (log I's mu_20 converges more slowly as v^2/x grows: up to 1e-13 inside
// log K's ranges).  Pairs of these ranges leave the power series and the K
// integral, the costliest expressions.
enum WideRanges { WIDE_NONE = 0, WIDE_I = 1, WIDE_K = 2 };
__device__ __forceinline__ bool tight_mu20_w(double v, double x, int w) {
  if (tight_mu20(v, x)) return true;
  if (w == WIDE_K)
    return (LB_GT(x, 18.5) && LB_LT(v, 9.5)) || (LB_GT(x, 20.0) && LB_LT(v, 12.5)) ||
           (LB_GT(x, 22.0) && LB_LT(v, 13.6));
  if (w == WIDE_I)
    return (LB_GT(x, 19.0) && LB_LT(v, 4.5)) || (LB_GT(x, 21.0) && LB_LT(v, 7.5)) ||
           (LB_GT(x, 23.0) && LB_LT(v, 9.5));
  return false;
}
__device__ __forceinline__ bool tight_u13_w(double v, double x, int w) {
  if (tight_u13(v, x)) return true;
  if (w == WIDE_K) return (LB_GT(x, 19.0) && LB_GT(v, 10.0)) || (LB_GT(x, 14.0) && LB_GT(v, 14.0));
  if (w == WIDE_I)
    return (LB_GT(x, 19.5) && LB_GT(v, 10.0)) || (LB_GT(x, 17.5) && LB_GT(v, 12.0)) ||
           (LB_GT(x, 14.5) && LB_GT(v, 14.0));
  return false;
}

// With the pairs binned per expression on chip (no warp divergence), the
// tight dispatch also uses the shorter uniform expansions of the paper's CPU
// order, with order thresholds from the same error map: U_4 for v > 230,
// U_6 for v > 70, U_9 for v > 28 (truncation <= 2e-16 for every x).
// w: WIDE_I or WIDE_K for values of log I or log K (K callers pass |v|),
// which take the wider mu_20 and U_13 ranges above; WIDE_NONE for the
// x-derivatives.
__device__ __forceinline__ int classify(double v, double x, int mode, int w = WIDE_NONE) {
  if (mode == MODE_TIGHT) {
    if (tight_mu20_w(v, x, w)) return R_MU20;
    if (LB_GT(v, 230.0)) return R_U4;
    if (LB_GT(v, 70.0)) return R_U6;
    if (LB_GT(v, 28.0)) return R_U9;
    if (tight_u13_w(v, x, w)) return R_U13;
    return R_FALLBACK;
  }
  if (mode == MODE_PAPER_CPU) {
    if (paper_mu3(v, x)) return R_MU3;
    if (paper_mu20(v, x)) return R_MU20;
    if (paper_u4(v, x)) return R_U4;
    if (paper_u6(v, x)) return R_U6;
    if (paper_u9(v, x)) return R_U9;
    if (paper_u13(v, x)) return R_U13;
    return R_FALLBACK;
  }
  if (paper_mu20(v, x)) return R_MU20;
  if (paper_u13(v, x)) return R_U13;
  return R_FALLBACK;
}

// ---------------------------------------------------------------------------
// mu_K expression (K terms after the leading 1):
//   S = 1 + sum_{k=1}^{K} s^k prod_{j<=k} (mu - (2j-1)^2) / (k! (8x)^k),  mu = 4v^2
//   log I = x - log(2 pi x)/2 + log|S|          (s = -1)
//   log K = log(pi / (2x))/2 - x + log|S|       (s = +1)
// S is formed by Horner's rule on the term ratios
//   r_k = (mu - (2k-1)^2) / (8 x k),  S = 1 + s r_1 (1 + s r_2 (1 + ... (1 + s r_K))).
// ---------------------------------------------------------------------------
// The number of terms actually summed is the smallest n <= K after which
// the terms fall below 2^-56 (a later term is then below the rounding of S);
// h is the first from which they are below 1e-3 (the leading h terms are
// summed in FP64, the rest in double-float).  Both depend on v^2/(2x) and
// 1/(8x) alone and come from a table over half octaves of the two
// (muterms_table.h, the largest of each cell): 15 instructions, where a pass
// over the 20 terms for each count took 160.  n averages 14.5 on the sweep's
// mu_20 pairs (13.7 exact).  Made uniform across the warp, so the Horner loop
// never diverges; the tile kernel orders the region by n while it bins the
// pairs, so the warps' lanes need similar counts.
#define LB_MUT_TABLE static __device__ const
#include "muterms_table.h"

// n | h << 8.
__device__ __forceinline__ int mu_counts(float v, float x) {
  const float w = __fdividef(1.0f, 8.0f * x), A = 4.0f * v * v * w;
  const int ia = (int)(__float_as_uint(A) >> 22) - LB_MUT_A_BASE, iw = (int)(__float_as_uint(w) >> 22) - LB_MUT_W_BASE;
  const int ca = ia < 0 ? 0 : (ia > LB_MUT_A_CELLS ? LB_MUT_A_CELLS : ia);
  const int cw = iw < 0 ? 0 : (iw > LB_MUT_W_CELLS ? LB_MUT_W_CELLS : iw);
  return (int)__ldg(lb_mut + cw * (LB_MUT_A_CELLS + 1) + ca);
}

// Terms of the power series of log I (series_log_i_n, series_so): the count
// n after which a term falls below 2^-56 of the running sum past the peak
// index (Eq. "K"), by a single-precision pass; at most 90.  Returned packed
// with the number h of leading terms kept in FP64: the terms past the peak
// from the first one below 1e-4 of the running sum on are summed in
// double-float (their part of the sum is below 1e-3 of it), as
// n + 128 h (series_count, series_head unpack it).
__device__ __forceinline__ int series_terms(float v, float x) {
  int n = 1, h = 0;
  const float yf = 0.25f * x * x;
  const float kpk = 0.5f * (sqrtf(fmaf(x, x, v * v)) - v);
  float term = 1.0f, T = 0.0f, kf = 0.0f;
#pragma unroll 1
  for (int k = 1; k <= 90; ++k) {
    kf += 1.0f;
    term *= __fdividef(yf, kf * (kf + v));         // an estimate: the fast division suffices
    T += term;
    n = k;
    if (h == 0 && kf > kpk && term <= 1e-4f * (1.0f + T)) h = k;
    if (kf > kpk && term <= 1.4e-17f * (1.0f + T)) break;
  }
  return n + 128 * (h == 0 ? n : h);
}
__device__ __forceinline__ int series_count(int packed) { return packed & 127; }
__device__ __forceinline__ int series_head(int packed) { return packed >> 7; }

// (2k-1)^2 for k = 1..20, and 20!/(k-1)! for k = 1..21 as doubles (exact) and
// as pairs of floats (entries 0 unused).
static __constant__ float kMuOdd[21] = {0.0f, 1.0f, 9.0f, 25.0f, 49.0f, 81.0f, 121.0f, 169.0f, 225.0f, 289.0f, 361.0f, 441.0f, 529.0f, 625.0f, 729.0f, 841.0f, 961.0f, 1089.0f, 1225.0f, 1369.0f, 1521.0f};
static __constant__ double kMuOddD[21] = {0.0, 1.0, 9.0, 25.0, 49.0, 81.0, 121.0, 169.0, 225.0, 289.0, 361.0, 441.0, 529.0, 625.0, 729.0, 841.0, 961.0, 1089.0, 1225.0, 1369.0, 1521.0};
static __constant__ double kMuF[22] = {0.0, 2432902008176640000.0, 2432902008176640000.0, 1216451004088320000.0, 405483668029440000.0, 101370917007360000.0, 20274183401472000.0, 3379030566912000.0, 482718652416000.0, 60339831552000.0, 6704425728000.0, 670442572800.0, 60949324800.0, 5079110400.0, 390700800.0, 27907200.0, 1860480.0, 116280.0, 6840.0, 380.0, 20.0, 1.0};
static __constant__ float kMuFd[22][2] = {{0.0f, 0.0f}, {2.4329020231636746e+18f, -14987034624.0f}, {2.4329020231636746e+18f, -14987034624.0f}, {1.2164510115818373e+18f, -7493517312.0f}, {4.054836705272791e+17f, -2497839104.0f}, {1.0137091763181978e+17f, -624459776.0f}, {2.0274182667370496e+16f, 734101504.0f}, {3379030623518720.0f, -56606720.0f}, {482718655709184.0f, -3293184.0f}, {60339831963648.0f, -411648.0f}, {6704425598976.0f, 129024.0f}, {670442586112.0f, -13312.0f}, {60949323776.0f, 1024.0f}, {5079110656.0f, -256.0f}, {390700800.0f, 0.0f}, {27907200.0f, 0.0f}, {1860480.0f, 0.0f}, {116280.0f, 0.0f}, {6840.0f, 0.0f}, {380.0f, 0.0f}, {20.0f, 0.0f}, {1.0f, 0.0f}};
constexpr long long kMuLogI = -760474846706970267ll;   // log(8/(2 pi)) - 2 log 20!, Q53
constexpr long long kMuLogK = -739853226357565351ll;   // log(4 pi) - 2 log 20!, Q53

// (log z + c) 2^53 for c in Q53: the fixed-point logarithm, or (z = 0,
// subnormal, infinite or NaN, as a forced evaluation far outside gives) the
// library's.
static __device__ __noinline__ double log_q53_plus(double z, long long c) {
  const uint32_t hi = (uint32_t)(ix_bits(z) >> 32);
  if (hi - 0x00100000u < 0x7fe00000u) return (double)(ix_log_q53(z) + c);
  return fma(log(z), 0x1p53, (double)c);
}

// mu_K with the lane's counts (mu_counts) given, at most cap terms; all 32
// lanes of the warp call it together.  20! S by Horner's rule without the
// divisions by k: with D_k = (mu - (2k-1)^2) s/(8x), Q <- D_k Q + 20!/(k-1)!
// from Q = 20!/n! down to k = 1.
template <int KIND>
__device__ __forceinline__ double mu_expr_n(double v, double x, int counts, int cap) {
  const int n = __reduce_max_sync(0xffffffffu, min(cap, counts & 255));
  const int h = min(n, __reduce_max_sync(0xffffffffu, counts >> 8));
  const double rx = ix_rcp_call(8.0 * x);                             // 1/(8x) on the integer pipe
  const double w = (KIND == KIND_I) ? -rx : rx;                       // the sign s folded in
  const double A = (4.0 * v * v) * w;
  double Q = kMuF[n + 1];
  if (n > h) {
    // terms h+1..n in double-float
    const dfloat wd = df_from_double(w), Ad = df_from_double(A);
    dfloat Qd = df_make(kMuFd[n + 1][0], kMuFd[n + 1][1]);
#pragma unroll 1
    for (int k = n; k > h; --k)
      Qd = df_mul_add(df_mulf_add(wd, -kMuOdd[k], Ad), Qd, df_make(kMuFd[k][0], kMuFd[k][1]));
    Q = df_to_double(Qd);
  }
#pragma unroll 1
  for (int k = h; k >= 1; --k) Q = fma(fma(-kMuOddD[k], w, A), Q, kMuF[k]);
  // log(S / sqrt(2 pi x)) = log(S^2 / (2 pi x)) / 2 and
  // log(S sqrt(pi / (2x))) = log(S^2 pi / (2x)) / 2, with 1/x = 8 rx: no
  // square root needed; the constants join the logarithm in Q53.
  return fma(0x1p-54, log_q53_plus(Q * Q * rx, KIND == KIND_I ? kMuLogI : kMuLogK), KIND == KIND_I ? x : -x);
}

// P_k(p) of the Debye polynomial u_k(t) = t^k P_k(t^2); k is a compile-time
// constant after unrolling, so the switch folds away.
template <typename T>
__device__ __forceinline__ T debye_P(int k, T p) {
  switch (k) {
    case 1: return lb_debye_P1(p);
    case 2: return lb_debye_P2(p);
    case 3: return lb_debye_P3(p);
    case 4: return lb_debye_P4(p);
    case 5: return lb_debye_P5(p);
    case 6: return lb_debye_P6(p);
    case 7: return lb_debye_P7(p);
    case 8: return lb_debye_P8(p);
    case 9: return lb_debye_P9(p);
    case 10: return lb_debye_P10(p);
    case 11: return lb_debye_P11(p);
    case 12: return lb_debye_P12(p);
    default: return lb_debye_P13(p);
  }
}

// P_k(p) in double-float, k = 2..13 (warp-uniform), by a rolled Horner
// loop over the coefficient pairs of lb_debye_df (constant memory, read by
// all lanes at once): the unrolled sums of U_13 alone would be about 1500
// instructions, and the tile kernel's warps run several expressions at a
// time out of one instruction cache.
__device__ __forceinline__ dfloat debye_P_df(int k, dfloat p) {
  const float(*c)[2] = lb_debye_df + lb_debye_df_off[k];
  dfloat r = df_make(c[k][0], c[k][1]);
#pragma unroll 1
  for (int i = k - 1; i >= 0; --i) r = df_mul_add(r, p, df_make(c[i][0], c[i][1]));
  return r;
}

// Q_k(p) in double-float, k = 2..13, from lb_debye_qdf (same layout).
__device__ __forceinline__ dfloat debye_Q_df(int k, dfloat p) {
  const float(*c)[2] = lb_debye_qdf + lb_debye_df_off[k];
  dfloat r = df_make(c[k][0], c[k][1]);
#pragma unroll 1
  for (int i = k - 1; i >= 0; --i) r = df_mul_add(r, p, df_make(c[i][0], c[i][1]));
  return r;
}

// ---------------------------------------------------------------------------
// U_K expression (paper Eqs. "log Iv u k", "log Kv u k"):
//   x' = x/v, r = sqrt(1 + x'^2), t = 1/r, eta = r + log(x' / (1 + r)),
//   S = 1 + sum_{k=1}^{K} (+-1)^k u_k(t) / v^k  (+ for I, alternating for K)
//   log I = -log(2 pi v)/2 + v eta - log(1 + x'^2)/4 + log|S|
//   log K =  log(pi/(2v))/2 - v eta - log(1 + x'^2)/4 + log|S|
// with u_k(t) = t^k P_k(t^2) (Debye polynomials, generated exactly from the
// recurrence of Eqs. "u0", "uk").  The two log terms are merged:
// -log(2 pi v)/2 - log(r)/2 = log(1 / sqrt(2 pi v r)).
// ---------------------------------------------------------------------------
// Evaluated by u_fx (lb_uniform.cuh) wherever r = sqrt(v^2 + x^2) lies in
// [16.04, 1e150] (every pair of the tight dispatch with v below that); this
// form serves the rest: the paper's U_13 from v = 12.7 on, forced
// evaluations, and extreme orders.
template <int KIND>
static __device__ __noinline__ double u_expr(double v, double x, int K) {
  const double inv_v = ix_rcp_call(v);           // reciprocal and root on the integer pipe
  const double xp = x * inv_v;
  double r, t;
  if (LB_LT(xp, 1e150)) {
    const double r2 = fma(xp, xp, 1.0);
    t = ix_rsqrt_call(r2);                       // t = (1 + x'^2)^-1/2
    r = r2 * t;
  } else {
    r = xp;                                      // 1 + x'^2 rounds to x'^2
    t = ix_rcp_call(r);
  }
  const double p = t * t;
  const double tq = t * inv_v;                    // t / v
  const double q = (KIND == KIND_K) ? -tq : tq;
  // Horner in q over k = K..1:  S = 1 + q (P_1 + q (P_2 + ... + q P_K)).
  // The terms k >= 2 (at most 1/v^2 of the sum, with v > 0.7 and x' > 35 or
  // v > 16 in the U regions: below 1e-3 of it) in double-float, P_1 and the
  // two outer steps in FP64.
  const dfloat pd = df_from_double(p), qd = df_from_double(q);
  dfloat accd = debye_P_df(K, pd);
#pragma unroll 1
  for (int k = K - 1; k >= 2; --k) accd = df_mul_add(accd, qd, debye_P_df(k, pd));
  const double acc = fma(df_to_double(accd), q, lb_debye_P1(p));
  const double S = fma(acc, q, 1.0);
  const double eta = r + (ix_log_call(xp) - ix_log_call(1.0 + r));      // log(x' / (1 + r)), no division
  // log(S / sqrt(2 pi v r)) = log(S^2 t / v) / 2 - log(2 pi) / 2, and for K
  // log(S sqrt(pi / (2 v r))) = log(S^2 t / v) / 2 + log(pi / 2) / 2
  // (t = 1/r): no root, and the constant joins the FMA with v eta.
  const double w = S * S * tq;
  if (KIND == KIND_I) return fma(0.5, ix_log_call(w), fma(v, eta, -kHalfLog2Pi));
  return fma(0.5, ix_log_call(w), fma(-v, eta, kHalfLogHalfPi));
}

// ---------------------------------------------------------------------------
// Power series of I_v (fallback region of log I):
//   a_0 = 1/Gamma(v+1), a_{k+1} = a_k x^2 / (4 (k+1)(k+v+1))      (Eq. "ak recurrence")
//   log I_v(x) = v log(x/2) + log a_0 + log sum_k a_k / a_0       (Eq. "log Iv")
// The log-sum-exp shift is a_0 instead of the peak term a_K: any shift is
// exact, and in the fallback region (x <= 30) the largest ratio a_K/a_0 is
// below e^x, far from overflow, so the terms can be summed in linear scale
// without a logarithm per term.  Terms are kept until they fall below 2^-56
// of the running sum after the peak index K = (-v + sqrt(x^2 + v^2))/2
// (Eq. "K"), the truncation rule of Sec. 3.1; the count n is found with a
// single-precision pass and made uniform across the warp.  The sum
//   S = 1 + r_1 (1 + r_2 (1 + ... (1 + r_n))),  r_k = y / (k (k + v)),  y = x^2/4,
// is then evaluated backwards as a fraction A/B (A <- d_k B + y A,
// B <- d_k B with d_k = k (k + v)), so the double-precision loop has no
// division; B stays below 1e250 for n <= 80 and v <= 16.  All 32 lanes of the
// warp must call it together.
// ---------------------------------------------------------------------------
// k and k^2 for k = 0, 1, ..., 90 as doubles (exact): the series loop reads
// them from constant memory (k is warp-uniform) and forms d_k = k (k + v) as
// one FMA, k v + k^2, instead of an addition and a multiplication.
static __constant__ double kSeriesK[91] = {
    0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16, 17, 18, 19, 20, 21, 22, 23, 24, 25,
    26, 27, 28, 29, 30, 31, 32, 33, 34, 35, 36, 37, 38, 39, 40, 41, 42, 43, 44, 45, 46, 47, 48, 49,
    50, 51, 52, 53, 54, 55, 56, 57, 58, 59, 60, 61, 62, 63, 64, 65, 66, 67, 68, 69, 70, 71, 72, 73,
    74, 75, 76, 77, 78, 79, 80, 81, 82, 83, 84, 85, 86, 87, 88, 89, 90};
static __constant__ double kSeriesK2[91] = {
    0, 1, 4, 9, 16, 25, 36, 49, 64, 81, 100, 121, 144, 169, 196, 225, 256, 289, 324, 361, 400, 441,
    484, 529, 576, 625, 676, 729, 784, 841, 900, 961, 1024, 1089, 1156, 1225, 1296, 1369, 1444,
    1521, 1600, 1681, 1764, 1849, 1936, 2025, 2116, 2209, 2304, 2401, 2500, 2601, 2704, 2809, 2916,
    3025, 3136, 3249, 3364, 3481, 3600, 3721, 3844, 3969, 4096, 4225, 4356, 4489, 4624, 4761, 4900,
    5041, 5184, 5329, 5476, 5625, 5776, 5929, 6084, 6241, 6400, 6561, 6724, 6889, 7056, 7225, 7396,
    7569, 7744, 7921, 8100};

// y / (k (k + v)) in double-float: the denominator from k v + k^2 (k^2
// exact), the quotient as q1 + q2 (Dekker: q1 from the leading parts, q2
// from the remainder y - q1 d).
__device__ __forceinline__ dfloat series_ratio_df(dfloat y, dfloat v, int k) {
  const float kf = (float)k;
  const dfloat d = df_add(df_mul(v, df_make(kf, 0.0f)), df_make(kf * kf, 0.0f));
  const float q1 = y.h * __frcp_rn(d.h);
  const dfloat rem = df_add(y, df_mul(d, df_make(-q1, 0.0f)));
  const float q2 = rem.h * __frcp_rn(d.h);
  dfloat r;
  r.h = q1 + q2;
  r.l = q2 - (r.h - q1);
  return r;
}

// lgamma(v + 1): lg_lgamma1p, or (orders past 17, as forced evaluations have)
// the library's.
static __device__ __noinline__ double lgamma1p(double v) { return lg_ok(v) ? lg_lgamma1p(v) : lgamma(v + 1.0); }

__device__ __forceinline__ double series_log_i_n(double v, double x, int packed) {
  const int n = __reduce_max_sync(0xffffffffu, series_count(packed));
  const int h = __reduce_max_sync(0xffffffffu, series_head(packed));
  const double y = 0.25 * x * x;
  double A = 1.0, B = 1.0;
  int top = n;
  if (n > h) {
    // terms h+1..n: P <- 1 + (y / (k (k + v))) P in double-float; its value
    // then starts the FP64 fraction (A / B = P)
    const dfloat yd = df_from_double(y), vd = df_from_double(v);
    dfloat Pd = df_make(1.0f, 0.0f);
#pragma unroll 1
    for (int k = n; k > h; --k) Pd = df_mul_add(series_ratio_df(yd, vd, k), Pd, df_make(1.0f, 0.0f));
    A = df_to_double(Pd);
    top = h;
  }
#pragma unroll 1
  for (int k = top; k >= 1; --k) {
    const double d = fma(kSeriesK[k], v, kSeriesK2[k]);   // k (k + v), exact up to one rounding
    A = fma(d, B, y * A);
    B *= d;
  }
  double res = ix_log_call(A * ix_rcp_call(B)) - lgamma1p(v);
  if ((__double_as_longlong(v) << 1) != 0) res = fma(v, ix_log_call(0.5 * x), res);   // v != 0, on the bits
  return res;
}

// ---------------------------------------------------------------------------
// One order for every argument (v_stride 0).  The order-dependent parts of
// the expressions are then the same for every pair, and a block computes
// them once (scalar_order_setup):
//   mu_K:   S = sum_k a_k w^k, w = 1/(8x), a_k = s^k prod_{j<=k} (mu - (2j-1)^2) / k!
//           -- one fixed-point multiply-add per term, no FP64, where that
//           keeps enough of S (lb_order.cuh);
//   series: P <- 1 + (y / (k (k + v))) P with the reciprocals 1/(k (k + v))
//           tabulated -- two operations per term instead of six, and
//           lgamma(v + 1) once.
// The sums are the same sums in another order of operations.
// ---------------------------------------------------------------------------
struct ScalarOrder {
  double v, lg1;                        // v, lgamma(v + 1)
  double scale;                         // so_scale
  bool mu_general;                      // so_general
  long long muc;                        // so_log_const and log(scale), Q53
  long long mu[21];                     // so_coef of b_0 .. b_20
  int uk;                               // so_u_terms
  long long u[40];                      // so_u_coef
  double ser[91];                       // 1 / (k (k + v)), k = 1..90
  dfloat serd[91];                      // ser[] in double-float
};

// All threads of the block (at least 64) call it; ends with a barrier.  The
// chains are kept short, as every block runs this before its first tile: the
// 20 ratios of mu_K on 20 lanes and their products by a warp scan, lgamma on
// another warp, the series' reciprocals on the rest.
template <int KIND, int NT>
__device__ __forceinline__ void scalar_order_setup(ScalarOrder& so, double v, int mode) {
  const int tid = threadIdx.x;
  if (tid < 32) {
    const int k = tid < 20 ? tid : 20;
    const double rf = __ldg(&lb_rfact[k][0]), rfl = __ldg(&lb_rfact[k][1]);
    const double scale = so_scale(KIND, mode == MODE_TIGHT, v);
    long long ls = ix_log_q53(scale);
    asm volatile("" : "+l"(ls));                    // here: its table reads wait beside the products
    double bl, b = so_ratio(KIND, v, k < 1 ? 1 : k, scale, bl);
    if (tid == 0) { b = 1.0; bl = 0.0; }
    if (so_pairs(v)) {
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {            // k! b_k, k = tid
        const double u = __shfl_up_sync(0xffffffffu, b, o), ul = __shfl_up_sync(0xffffffffu, bl, o);
        if (tid >= o) so_mul(b, bl, u, ul);
      }
      so_mul(b, bl, rf, rfl);
    } else {
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, b, o);
        if (tid >= o) b *= u;
      }
      b *= rf;
      bl = 0.0;
    }
    const int muq = __reduce_max_sync(0xffffffffu, tid <= 20 ? so_size(b) : 0);
    if (tid <= 20) so.mu[tid] = so_coef(b, bl, muq);
    if (tid == 0) {
      so.v = v;
      so.scale = scale;
      so.mu_general = so_general(KIND, muq, scale);
      so.muc = so_log_const(KIND, muq) + ls;
    }
  } else if (tid < 64) {
    if (tid == 32) so.lg1 = lgamma1p(v);
  }
  static_assert(NT >= 256, "warps for every part");
  if (tid >= 64 && tid < 154) {
    const int k = tid - 63;
    so.ser[k] = 1.0 / ((double)k * ((double)k + v));
    so.serd[k] = df_from_double(so.ser[k]);
  } else if (tid >= 160 && tid < 200) {
    const int K = so_u_terms(v, mode), m = tid - 160;
    if (m <= 3 * K) so.u[m] = so_u_coef(KIND, v, K, m, lb_debye_c);
    if (m == 0) so.uk = K;
  }
  __syncthreads();
}

template <int KIND>
__device__ __forceinline__ double mu_expr_so(const ScalarOrder& so, double x, int counts) {
  if (KIND == KIND_I && so.mu_general) return mu_expr_n<KIND>(so.v, x, counts, 20);   // the same for the whole block
  const int n = __reduce_max_sync(0xffffffffu, counts & 255);
  const double W = ix_rcp_call(so.scale * x);
  const double S = so_sum(so.mu, W, n);
  return fma(0x1p-54, log_q53_plus(S * S * W, so.muc), KIND == KIND_I ? x : -x);
}

__device__ __forceinline__ double series_so(const ScalarOrder& so, double x, int packed) {
  const double v = so.v;
  const int n = __reduce_max_sync(0xffffffffu, series_count(packed));
  const int h = __reduce_max_sync(0xffffffffu, series_head(packed));
  const double y = 0.25 * x * x;
  double P = 1.0;
  int top = n;
  if (n > h) {                                    // terms h+1..n in double-float
    const dfloat yd = df_from_double(y);
    dfloat Pd = df_make(1.0f, 0.0f);
#pragma unroll 1
    for (int k = n; k > h; --k) Pd = df_mul_add(df_mul(yd, so.serd[k]), Pd, df_make(1.0f, 0.0f));
    P = df_to_double(Pd);
    top = h;
  }
#pragma unroll 1
  for (int k = top; k >= 1; --k) P = fma(y * so.ser[k], P, 1.0);
  double res = ix_log_call(P) - so.lg1;
  if ((__double_as_longlong(v) << 1) != 0) res = fma(v, ix_log_call(0.5 * x), res);   // v != 0, on the bits
  return res;
}

// ---------------------------------------------------------------------------
// x-derivatives of the same expressions (the adjoint of the forward path).
// Each differentiates its expression term by term, so it is valid exactly
// where the expression is; the paper lists derivatives as future work
// (Sec. 7), and these follow directly from its Eqs.
// ---------------------------------------------------------------------------

// mu_K: log f = +-x - log(2 pi x)/2 + log S (I: +x, K: -x and +log(pi/2)/2),
// S = 1 + sum_k c_k w^k, w = 1/(8x), so with E = w dS/dw
//   d/dx log f = +-1 - (1/x) (1/2 + E/S).
// The sums as mu_expr_n's: Q <- D_k Q + 20!/(k-1)! and, D_k being
// proportional to w, R <- D_k (Q + R) beside it; the terms past the leading
// h in double-float, at most cap terms.  For half an odd integer the sum ends
// (D_(v + 1/2) = 0): order 1/2, 5M pairs, x in [1, 100], 575 -> 512 us.
template <int KIND>
__device__ __forceinline__ double mu_dx_n(double v, double x, int counts, int cap) {
  {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v), M = (b & 0xfffffffffffffull) | (1ull << 52);
    const int p = 1074 - (int)(b >> 52);            // 2v = M / 2^p
    if (__ffsll((long long)M) - 1 == p) cap = min(cap, (int)(((M >> p) - 1) >> 1));
  }
  const int n = __reduce_max_sync(0xffffffffu, min(cap, counts & 255));
  const int h = min(n, __reduce_max_sync(0xffffffffu, counts >> 8));
  const double rx = ix_rcp_call(8.0 * x);           // on the integer pipe
  const double w = (KIND == KIND_I) ? -rx : rx;      // the sign folded in
  const double A = (4.0 * v * v) * w;
  double Q = kMuF[n + 1], R = 0.0;
  if (n > h) {
    const dfloat wd = df_from_double(w), Ad = df_from_double(A);
    dfloat Qd = df_make(kMuFd[n + 1][0], kMuFd[n + 1][1]), Rd = df_make(0.0f, 0.0f);
#pragma unroll 1
    for (int k = n; k > h; --k) {
      const dfloat D = df_mulf_add(wd, -kMuOdd[k], Ad);
      Rd = df_mul(D, df_add(Qd, Rd));
      Qd = df_mul_add(D, Qd, df_make(kMuFd[k][0], kMuFd[k][1]));
    }
    Q = df_to_double(Qd);
    R = df_to_double(Rd);
  }
#pragma unroll 1
  for (int k = h; k >= 1; --k) {
    const double D = fma(-kMuOddD[k], w, A);
    R = D * (Q + R);
    Q = fma(D, Q, kMuF[k]);
  }
  const double base = (KIND == KIND_I) ? 1.0 : -1.0;
  return base - (8.0 * rx) * fma(R, ix_rcp_call(Q), 0.5);
}

// U_K: with x' = x/v, t = (1 + x'^2)^-1/2, d(v eta)/dx = 1/(t x'),
// d/dx [-log(1 + x'^2)/4] = -x' t^2 / (2v), dt/dx = -x' t^3 / v and
// d/dt u_k(t) = t^(k-1) Q_k(t^2):
//   d/dx log f = +-1/(t x') - (x' t^2 / v) (1/2 + SQ / S),
//   S = 1 + sum q^k P_k(t^2), SQ = sum q^k Q_k(t^2), q = +-t/v.
// Evaluated by u_dx_fx (lb_uniform.cuh) wherever u_fx serves the values; this
// form for the rest.  K: the pair's own terms.
template <int KIND>
static __device__ __noinline__ double u_dx(double v, double x, int K) {
  const double inv_v = ix_rcp(v);                  // reciprocals and 1/sqrt on the integer pipe
  const double xp = x * inv_v;
  double r, t;
  if (xp < 1e150) {
    const double w = fma(xp, xp, 1.0);
    t = ix_rsqrt(w);
    r = w * t;
  } else {
    r = xp;
    t = ix_rcp(xp);
  }
  const double p = t * t;
  double q = t * inv_v;
  if (KIND == KIND_K) q = -q;
  // Horner in q over k = K..1 for S and SQ; as in u_expr, the terms k >= 2
  // (at most 1/v^2 of each sum in the U regions) in double-float, rolled
  // over the coefficient tables, and k = 1 and the outer steps in FP64.
  const dfloat pd = df_from_double(p), qd = df_from_double(q);
  dfloat aP = debye_P_df(K, pd), aQ = debye_Q_df(K, pd);
#pragma unroll 1
  for (int k = K - 1; k >= 2; --k) {
    aP = df_mul_add(aP, qd, debye_P_df(k, pd));
    aQ = df_mul_add(aQ, qd, debye_Q_df(k, pd));
  }
  const double accP = fma(df_to_double(aP), q, lb_debye_P1(p));
  const double accQ = fma(df_to_double(aQ), q, lb_debye_Q1(p));
  const double S = fma(accP, q, 1.0);
  const double SQ = accQ * q;
  const double lead = r * ix_rcp(xp);               // 1/(t x') = sqrt(1 + x'^2)/x'
  const double corr = (xp * p * inv_v) * fma(SQ, ix_rcp(S), 0.5);
  return (KIND == KIND_I) ? lead - corr : -lead - corr;
}

// Series: log I = v log(x/2) - lgamma(v+1) + log(1 + T), T = sum_{k>=1} a_k/a_0
// with a_k/a_0 proportional to x^(2k):  d/dx log I = v/x + (2/x) (sum k a_k/a_0) / (1 + T).
// With the pair's term count (series_terms): T and D = sum k a_k/a_0 by one
// backward Horner pass, P <- 1 + r_k P and E <- r_k (P + E) (E collects
// y dP/dy = D, as r_k is proportional to y), r_k = y / (k (k + v)); the
// terms past the head in double-float (as series_log_i_n), the head as one
// fraction P = A/B, E = C/B with A <- d B + y A, C <- y (A + C), B <- d B
// (d = k (k + v)), so no term divides; D/(1+T) = C/A.
__device__ __forceinline__ double series_dx_n(double v, double x, int packed) {
  const int n = __reduce_max_sync(0xffffffffu, series_count(packed));
  const int h = __reduce_max_sync(0xffffffffu, series_head(packed));
  const double y = 0.25 * x * x;
  double A = 1.0, C = 0.0, B = 1.0;
  int top = n;
  if (n > h) {
    const dfloat yd = df_from_double(y), vd = df_from_double(v);
    dfloat Pd = df_make(1.0f, 0.0f), Ed = df_make(0.0f, 0.0f);
#pragma unroll 1
    for (int k = n; k > h; --k) {
      const dfloat r = series_ratio_df(yd, vd, k);
      Ed = df_mul(r, df_add(Pd, Ed));
      Pd = df_mul_add(r, Pd, df_make(1.0f, 0.0f));
    }
    A = df_to_double(Pd);
    C = df_to_double(Ed);
    top = h;
  }
#pragma unroll 1
  for (int k = top; k >= 1; --k) {
    const double d = fma(kSeriesK[k], v, kSeriesK2[k]);   // k (k + v)
    C = y * (A + C);
    A = fma(d, B, y * A);
    B *= d;
  }
  return fma(2.0 * C, ix_rcp(A), v) * ix_rcp(x);
}

}  // namespace lb
