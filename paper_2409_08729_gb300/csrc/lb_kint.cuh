// lb_kint.cuh -- warp-cooperative evaluation of the K integral in the paper's
// form (device code; the paper's dispatches).
//
// Paper Sec. 3.2, Eq. "log Kv integral" (Rothwell's representation):
//   log K_v(x) = log(pi)/2 - lgamma(v + 1/2) - v log(2x) - x
//              + log int_0^1 [g(u) + h(u)] du,
//   g(u) = beta exp(-u^beta) (2x + u^beta)^(v-1/2) u^(n-1),  beta = 2n/(2v+1), n = 8,
//   h(u) = exp(-1/u) u^(-2v-1) (2xu + 1)^(v-1/2).
// One warp evaluates one pair: its lanes split the nodes of a composite
// Simpson rule on u in [0, 1], N = 600, with weights 4 (odd k), 2 (even k),
// 1 (k = N), the constant read as 1/(3N), f(0) = 0, and the paper's heuristic
// maxima log g(1) and log h(u*), u* = 1/2 (v < 2) or 1/(2v), as log-sum-exp
// shifts.  The tight mode takes the integral of lb_ktrap.cuh instead, one
// pair per thread.
#pragma once

#include "lb_expr.cuh"
#include "lb_intmath.cuh"

namespace lb {

__device__ __forceinline__ double warp_sum(double a) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}

// log of the prefactor sqrt(pi) e^{-x} / (Gamma(v+1/2) (2x)^v)
__device__ __forceinline__ double kint_prefactor(double v, double x) {
  return kHalfLogPi - lgamma(v + 0.5) - fma(v, ix_log(2.0 * x), x);
}

// Warp-cooperative log int_0^1 (g + h) du by the paper's Simpson rule (N = 600).
__device__ __forceinline__ double kint_log_simpson(double v, double x, int lane) {
  const int N = 600;
  const double beta = 16.0 / (2.0 * v + 1.0);
  const double logbeta = log(beta);
  const double vm = v - 0.5, tx = 2.0 * x;
  const double a2 = 2.0 * v + 1.0;
  // heuristic maxima: g at u = 1, h at u* = 1/2 (v < 2) or 1/(2v)
  const double mg = logbeta - 1.0 + vm * log(tx + 1.0);
  const double us = (v < 2.0) ? 0.5 : 0.5 / v;
  const double mh = -1.0 / us - a2 * log(us) + vm * log1p(tx * us);
  double sg = 0.0, sh = 0.0;
  for (int k = lane + 1; k <= N; k += 32) {
    const double u = (double)k / (double)N;
    const double w = (k == N) ? 1.0 : ((k & 1) ? 4.0 : 2.0);
    const double lu = log(u);
    const double ub = exp(beta * lu);
    const double lg = logbeta - ub + fma(vm, log(tx + ub), 7.0 * lu);
    const double lh = -1.0 / u - a2 * lu + vm * log1p(tx * u);
    sg = fma(w, exp(lg - mg), sg);
    sh = fma(w, exp(lh - mh), sh);
  }
  sg = warp_sum(sg);
  sh = warp_sum(sh);
  const double lG = mg + log(sg), lH = mh + log(sh);
  const double M = fmax(lG, lH);
  return M + log(exp(lG - M) + exp(lH - M)) - log(3.0 * N);
}

}  // namespace lb
