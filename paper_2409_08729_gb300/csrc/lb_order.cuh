// lb_order.cuh -- expansions of a call whose pairs all have one order, in fixed
// point: mu_20 (here) and U_K (below).
//
// With one order mu_20's sum is a polynomial in 1/x with constant coefficients,
// S = sum_k a_k / (8x)^k, a_k = s^k prod_{j<=k} (mu - (2j-1)^2) / k!: one integer
// multiply-add per term.  In W = xmin / (2x), xmin the smallest x at which the
// dispatch takes mu_20 for the order, the coefficients are b_k = a_k /
// (4 xmin)^k, and with muq the exponent of the largest of them the sums are
// kept in Q(60 - muq): as W <= 1/2, every Horner sum stays within +-2^62, and S
// is within 2^(muq - 58) (a truncation and a coefficient's rounding per step,
// halved by the next).
//
// That is an absolute bound, and log I's S is small where v^2/(2x) is large
// (about exp(-v^2/(2x)), down to 0.05), so muq has to be small: hence the scale
// by xmin itself.  muq is then at most 5 in tight mode; one power of two for
// all orders below 15.4 left it at 11 to 14 for orders from 13 on and log I up
// to 5.3e-15 off (v = 13.59, x = 30.1; now 3.3e-16, the expansion's truncation
// included).  Where it is above 6 all the same (the paper's dispatch, log I,
// orders about 15, x from 30 on) the general form serves (so_general).
//
// The functions compile for the host too (without __CUDACC__).
#pragma once

#include "lb_intmath.cuh"
#include "lb_ktrap.cuh"
#include "lb_uniform.cuh"

namespace lb {

constexpr long long kSoLogI56 = -132432999542942538ll, kSoLogK56 = 32539963252296791ll;   // -log(2 pi), log(pi/2), Q56
constexpr long long kLn2Q56 = 49946518145322874ll;

// 1/k! as pairs of doubles, k = 0 .. 20.
LB_IX_TABLE double lb_rfact[21][2] = {
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.0000000000000p+0, 0x0.0p+0},
    {0x1.0000000000000p-1, 0x0.0p+0}, {0x1.5555555555555p-3, 0x1.5555555555555p-57},
    {0x1.5555555555555p-5, 0x1.5555555555555p-59}, {0x1.1111111111111p-7, 0x1.1111111111111p-63},
    {0x1.6c16c16c16c17p-10, -0x1.f49f49f49f49fp-65}, {0x1.a01a01a01a01ap-13, 0x1.a01a01a01a01ap-73},
    {0x1.a01a01a01a01ap-16, 0x1.a01a01a01a01ap-76}, {0x1.71de3a556c734p-19, -0x1.c154f8ddc6c00p-73},
    {0x1.27e4fb7789f5cp-22, 0x1.cbbc05b4fa99ap-76}, {0x1.ae64567f544e4p-26, -0x1.c062e06d1f209p-80},
    {0x1.1eed8eff8d898p-29, -0x1.2aec959e14c06p-83}, {0x1.6124613a86d09p-33, 0x1.f28e0cc748ebep-87},
    {0x1.93974a8c07c9dp-37, 0x1.05d6f8a2efd1fp-92}, {0x1.ae7f3e733b81fp-41, 0x1.1d8656b0ee8cbp-97},
    {0x1.ae7f3e733b81fp-45, 0x1.1d8656b0ee8cbp-101}, {0x1.952c77030ad4ap-49, 0x1.ac981465ddc6cp-103},
    {0x1.6827863b97d97p-53, 0x1.eec01221a8b0bp-107}, {0x1.2f49b46814157p-57, 0x1.2650f61dbdcb4p-112},
    {0x1.e542ba4020225p-62, 0x1.ea72b4afe3c2fp-120},
};

// Argument scale 2 / xmin: W = 1 / (scale x).  xmin as the dispatches have it
// (classify), at the curved edges with room for their single precision, at
// most 1e290 (there x is larger still).  No division: every block waits for it.
LB_IX_FN double so_scale(int kind, bool tight, double v) {
  constexpr double kRoom = 1.0 + 0x1p-40;                   // W below 1/2 after its rounding too
  if (v < (tight ? 13.6 : 15.3919)) {
    if (!tight) return kRoom * 2.0 / 30.0;
    if (kind == 0) return v < 4.5 ? kRoom * 2.0 / 19.0 : v < 7.5 ? kRoom * 2.0 / 21.0
                        : v < 9.5 ? kRoom * 2.0 / 23.0 : kRoom * 2.0 / 30.0;
    return v < 9.5 ? kRoom * 2.0 / 18.5 : v < 12.5 ? kRoom * 2.0 / 20.0 : kRoom * 2.0 / 22.0;
  }
  double m = v * v * ((1.0 - 1e-5) / 6.48);                 // xmin / 2: v^2 < 3.24 x
  if (!tight) {                                             // 0.5113 log x + 0.7939 > log v: x > (v/2.212)^1.9558
    const int e = v < 1e300 ? ilogb(v) : 1000;
    const float l = 1.9558f * ((float)e + log2f((float)scalbn(v, -e)) - 1.1454f);
    const float f = floorf(l);
    m = fmin(m, scalbn((double)exp2f(l - f), (int)f) * 0.4995);
  }
  return ix_rcp(fmin(fmax(m, 29.845), 1e290));
}

// k b_k / b_(k-1), k = 1 .. 20, as a sum hi + lo.
LB_IX_FN double so_ratio(int kind, double v, int k, double scale, double& lo) {
  const double odd = (double)((2 * k - 1) * (2 * k - 1)), c = (kind == 0 ? -0.125 : 0.125) * scale, t = 2.0 * v;
  const double m = t * t, ml = fma(t, t, -m), d = m - odd;
  const double dl = (m >= odd ? (m - d) - odd : m - (odd + d)) + ml;   // d + dl = 4 v^2 - odd
  const double p = d * c;
  lo = fma(dl, c, fma(d, c, -p));
  return p;
}

// Whether the coefficients are formed as pairs of doubles: where log I's S is
// 0.02 to 0.1 (orders from 11.5 to 15.4, x about 30) the terms reach 5, and
// coefficients rounded to doubles would cost log S 20 roundings (order 13.59:
// mean error 2.4e-16 of the result, 0.4e-16 with the pairs).  Elsewhere log I's S is
// above 0.08 and both give the same errors; the pairs would cost every block
// 0.9 us.
LB_IX_FN bool so_pairs(double v) { return v >= 11.5 && v < 15.4; }

// (b + bl) <- (b + bl) (u + ul)
LB_IX_FN void so_mul(double& b, double& bl, double u, double ul) {
  const double p = b * u;
  bl = fma(bl, u, fma(b, ul, fma(b, u, -p)));
  b = p;
}

// One coefficient's part of muq (the largest of them counts, at most 50).
LB_IX_FN int so_size(double b) {
  if (b == 0.0) return 0;
  const int e = ilogb(fabs(b));
  return e < 0 ? 0 : (e > 50 ? 50 : e);
}

// Whether mu_20 takes the general form for this order.  Above xmin = 2^14 the
// size of x itself makes any such error small.
LB_IX_FN bool so_general(int kind, int muq, double scale) { return kind == 0 && muq > 6 && scale > 0x1p-13; }

// b_k in Q(60 - muq), plus 2^62 (nothing where it overflows: orders past 1e150,
// whose x is so large that only the leading 1 counts).
LB_IX_FN long long so_coef(double b, double bl, int muq) {
  if (!(fabs(b) < 0x1p51)) return 1ll << 62;
  return ix_fix(b, 60 - muq) + ix_fix(bl, 60 - muq) + (1ll << 62);
}

// The logarithm's constant less log(scale), Q53: with 1/x = scale W,
// log I = x + (log((S 2^(60 - muq))^2 W) + it + log(scale)) / 2.
LB_IX_FN long long so_log_const(int kind, int muq) {
  return ((kind == 0 ? kSoLogI56 : kSoLogK56) - 2 * (60 - muq) * kLn2Q56 + 4) >> 3;
}

// S 2^(60 - muq) by Horner's rule, n terms past the first; W = 1/(scale x).  On
// the sums plus 2^62 (from 0 to 2^63: the short unsigned product), the bias's
// product taken off again.  Unrolled by 4: order 8, 20M pairs, 871 us by 2, 862
// by 4.
LB_IX_FN double so_sum(const long long* b, double W, int n) {
  const uint64_t w = (uint64_t)ix_fix(W, 64);              // below 2^63
  const uint64_t bias = w >> 2;
  uint64_t acc = (uint64_t)b[n];
#if defined(__CUDACC__)
#pragma unroll 4
#endif
  for (int k = n - 1; k >= 0; --k) acc = (uint64_t)b[k] + kt_mulhi(acc, w) - bias;
  return (double)(long long)(acc - (1ull << 62));
}

// ---------------------------------------------------------------------------
// U_K of one order: with t = v/r, S = sum_k u_k(t) / (+-v)^k is one polynomial of
// degree 3K in t with constant coefficients, a multiply-add per power, where the
// sums over pairs (lb_uniform.cuh) take two for every second power of every
// term, and loops around them.  Built where one K serves the order (tight mode
// and the paper's GPU dispatch) and the order is above 10, so that the
// coefficients are below 1 and their sum below 1.6.  log I, 5M pairs, x in
// [1, 100]: order 14 366 -> 302 us, 20 460 -> 345, 40 389 -> 299, 300 271 -> 245;
// order 8, which has no U_K pairs there, unchanged.
// ---------------------------------------------------------------------------
// K, or 0: no polynomial for this order (mode: MODE_TIGHT 0, MODE_PAPER_GPU 1).
LB_IX_FN int so_u_terms(double v, int mode) {
  if (!(v > 10.0 && v < 1e150) || mode > 1) return 0;
  return mode == 1 ? 13 : v > 230.0 ? 4 : v > 70.0 ? 6 : v > 28.0 ? 9 : 13;
}

// The coefficient of t^m in Q61; c[k][i]: that of t^(k + 2i) in u_k.  The terms
// are k = m, m - 2, .. (at most K) down to m/3, five of them at most: Horner's
// rule in 1/v^2, then the lowest power of 1/v (a short chain: every block waits
// for it).
LB_IX_FN long long so_u_coef(int kind, double v, int K, int m, const double (*c)[14]) {
  const double iv = kind == 0 ? ix_rcp(v) : -ix_rcp(v), w = iv * iv;
  int k1 = m < K ? m : K, k0 = (m + 2) / 3;
  k1 -= (k1 ^ m) & 1;
  k0 += (k0 ^ m) & 1;
  double sum = 0.0;
#if defined(__CUDACC__)
#pragma unroll
#endif
  for (int j = 0; j < 5; ++j) {
    const int k = k1 - 2 * j;
    if (k >= k0) sum = fma(sum, w, c[k][(m - k) >> 1]);
  }
  double q = iv;
#if defined(__CUDACC__)
#pragma unroll
#endif
  for (int j = 0; j < 4; ++j) {                             // sum iv^k0, k0 <= 13
    if ((k0 >> j) & 1) sum *= q;
    q *= q;
  }
  return ix_fix(sum, 61);
}

// log I or log K from the polynomial's degree M and coefficients; s = v^2 + x^2, uni_ok.
LB_IX_FN double so_u(int kind, const long long* c, int M, double v, double x, double s) {
  const double q = kt_rsqrt(s), r = s * q;
  const uint64_t t = (uint64_t)ix_fix(v * q, 63);          // at most 2^63 (1 + 2^-52)
  // Horner on the sums plus 2^62 (between 0 and 2^63, the short product), the bias's product taken off
  const uint64_t off = (1ull << 62) - (t >> 1);
  uint64_t acc = (uint64_t)c[M] + (1ull << 62);
#if defined(__CUDACC__)
#pragma unroll 2
#endif
  for (int m = M - 1; m >= 0; --m) acc = (uint64_t)c[m] + off + (kt_mulhi(acc, t) << 1);
  return uni_log(kind, v, x, r, q, (acc - (1ull << 62)) << 1);
}

}  // namespace lb
