"""mu_20 and U_K of a call with one order (csrc/lb_order.cuh): the host build of
the block's set-up and of the fixed-point sums, over the orders at which a
scale, a degree or the form changes, in both dispatches.

The sum against the exact (rational) one: within 2^(muq - 58) absolute.  log I
in tight mode: muq <= 5 and S >= 0.048 (order 13.59 at x = 30), so 2.3e-15
relative against a result of the size of x >= 30, 0.8e-16 x; the rounding of W
moves S by v^2/(2x) <= 3.7 times 2^-52, 0.3e-16 x.  log K: smaller, S >= 0.9
where v is small and above 1 where muq is not 0.  The paper's dispatch: muq <= 6
in this form, S >= 0.027: 1.7e-16 x.  Bound taken: 2e-16 x.
The values against the oracle, in units of the error metric: the expansion's
truncation 3.1e-16, the sum 2e-16, logarithm and roundings 2.3e-16: 1e-15.
U_K's polynomial: truncation 4e-16, the sum 2^-54, its three logarithms (2^-53
each, times v) 2.2e-16, two roundings of the result 2.2e-16: 1e-15."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

import oracle

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_08729_gb300", "csrc")
TOL = 1e-15
SRC = r'''
#define __constant__
#define __host__
#define __device__
#define __forceinline__ inline
template <typename T> T lb_fma(T a, T b, T c);
#include "lb_df.cuh"
#include "debye_uk.h"
#include "lb_order.cuh"
#define LB_MUT_TABLE static const
#include "muterms_table.h"
using namespace lb;
// returns muq | general << 8; S (scaled back), the largest W, log I or log K, terms
extern "C" int order(int kind, int tight, double v, const double* x, double* S, double* f, int* terms, long n, double* Wmax) {
  const double scale = so_scale(kind, tight != 0, v);
  *Wmax = 0.0;
  double b[32], l[32], c[32], d[32];
  for (int t = 0; t < 32; ++t) b[t] = so_ratio(kind, v, t < 1 ? 1 : (t > 20 ? 20 : t), scale, l[t]);
  b[0] = 1.0;
  l[0] = 0.0;
  for (int o = 1; o < 32; o <<= 1) {                       // the warp's scan
    for (int t = 0; t < 32; ++t) { c[t] = b[t]; d[t] = l[t]; }
    for (int t = o; t < 32; ++t) {
      if (so_pairs(v)) so_mul(b[t], l[t], c[t - o], d[t - o]);
      else b[t] *= c[t - o];
    }
  }
  for (int t = 0; t <= 20; ++t) {
    if (so_pairs(v)) so_mul(b[t], l[t], lb_rfact[t][0], lb_rfact[t][1]);
    else { b[t] *= lb_rfact[t][0]; l[t] = 0.0; }
  }
  int muq = 0;
  for (int t = 0; t <= 20; ++t) muq = so_size(b[t]) > muq ? so_size(b[t]) : muq;
  long long mu[21];
  for (int t = 0; t <= 20; ++t) mu[t] = so_coef(b[t], l[t], muq);
  for (long i = 0; i < n; ++i) {
    const float w = 1.0f / (8.0f * (float)x[i]), A = 4.0f * (float)v * (float)v * w;
    const int ia = (int)(ix_fbits(A) >> 22) - LB_MUT_A_BASE, iw = (int)(ix_fbits(w) >> 22) - LB_MUT_W_BASE;
    const int ca = ia < 0 ? 0 : (ia > LB_MUT_A_CELLS ? LB_MUT_A_CELLS : ia);
    const int cw = iw < 0 ? 0 : (iw > LB_MUT_W_CELLS ? LB_MUT_W_CELLS : iw);
    terms[i] = lb_mut[cw * (LB_MUT_A_CELLS + 1) + ca] & 255;
    const double W = ix_rcp(scale * x[i]), s = so_sum(mu, W, terms[i]);
    *Wmax = fmax(*Wmax, W);
    S[i] = ldexp(s, muq - 60);
    f[i] = fma(0x1p-54, (double)(ix_log_q53(s * s * W) + so_log_const(kind, muq) + ix_log_q53(scale)), kind == 0 ? x[i] : -x[i]);
  }
  return muq | (int)so_general(kind, muq, scale) << 8;
}
// returns K; the values, and the largest of the coefficients past the first
extern "C" int poly(int kind, int mode, double v, const double* x, double* f, long n, double* cmax) {
  const int K = so_u_terms(v, mode);
  long long c[40];
  *cmax = 0.0;
  for (int m = 0; m <= 3 * K && K; ++m) {
    c[m] = so_u_coef(kind, v, K, m, lb_debye_c);
    if (m) *cmax = fmax(*cmax, fabs((double)c[m] * 0x1p-61));
  }
  for (long i = 0; i < n && K; ++i) f[i] = so_u(kind, c, 3 * K, v, x[i], fma(v, v, x[i] * x[i]));
  return K;
}
'''


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    d = tmp_path_factory.mktemp("order")
    src, so = str(d / "o.cpp"), str(d / "o.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-o", so, src],
                   check=True)
    L = ctypes.CDLL(so)

    def run(kind, tight, v, x):
        S, f, t = np.empty_like(x), np.empty_like(x), np.empty(x.size, dtype=np.int32)
        W = ctypes.c_double()
        r = L.order(kind, int(tight), ctypes.c_double(v), *(a.ctypes.data_as(ctypes.c_void_p) for a in (x, S, f, t)),
                    ctypes.c_long(x.size), ctypes.byref(W))
        return S, f, t, W.value, r & 255, bool(r >> 8)
    run.poly = L.poly
    return run


def _xmin(kind, tight, v):
    """The smallest x at which the dispatch takes mu_20."""
    if not tight:
        if v < 15.3919:
            return 30.0
        return max(59.6925, np.exp((np.log(v) - 0.7939) / 0.5113))
    if v >= 13.6:
        return max(59.6925, v * v / 3.24)
    if kind == 0:
        return 19.0 if v < 4.5 else 21.0 if v < 7.5 else 23.0 if v < 9.5 else 30.0
    return 18.5 if v < 9.5 else 20.0 if v < 12.5 else 22.0


_EDGES = [4.5, 7.5, 9.5, 12.5, 13.6, 15.3919]
ORDERS = sorted([0.0, 1e-300, 0.3, 2.5, 8.0, 10.5, 10.8, 10.9, 11.0, 12.0, 12.6964, 13.3, 13.59, 14.5, 15.0, 15.39, 16.0,
                 17.0, 20.0, 28.0, 40.0, 300.0, 1e4] + _EDGES + [np.nextafter(e, 0) for e in _EDGES])


@pytest.mark.parametrize("tight", [True, False])
@pytest.mark.parametrize("kind", [0, 1])
def test_sum_against_the_exact_sum(order, kind, tight):
    for v in ORDERS:
        x0 = _xmin(kind, tight, v)
        x = x0 * (1.0 + np.concatenate([[1e-9, 1e-3, 0.01, 0.05], np.geomspace(0.1, 30.0, 20)]))
        S, _, terms, W, muq, general = order(kind, tight, v, x)
        assert 0.49 < W < 0.5, v
        assert muq <= (6 if kind == 0 else 8) or (general and not tight) or x0 > 2.0 ** 14, (v, muq)
        if general:
            continue
        for xi, si, n in zip(x, S, terms):
            w = 1 / (8 * Fraction(float(xi)))
            s, t = Fraction(1), Fraction(1)
            for k in range(1, int(n) + 1):
                t *= (-1 if kind == 0 else 1) * (4 * Fraction(float(v)) ** 2 - (2 * k - 1) ** 2) * w / k
                s += t
            assert abs(float(Fraction(float(si)) / s - 1)) <= 2e-16 * xi, (v, xi, float(s), muq)


@pytest.mark.parametrize("kind", [0, 1])
def test_values_against_oracle(order, kind):
    r = np.random.default_rng(7)
    for v in ORDERS + list(r.uniform(0.0, 40.0, 40)):
        x0 = _xmin(kind, True, v) * (1 + 1e-9)
        x = x0 * np.concatenate([1.0 + 0.1 * r.random(150), np.exp(3.0 * r.random(150))])
        x = x[x < 1e8]                                # the oracle's power series stops there
        _, f, _, _, _, general = order(kind, True, v, x)
        assert not general
        vv = np.full_like(x, v)
        ref = (oracle.log_k if kind else oracle.log_i)(vv, x)
        err = oracle.rel_err(f, ref, oracle.error_scale("ik"[kind], vv, x))
        assert err.max() <= TOL, (v, x[err.argmax()], err.max())


@pytest.mark.parametrize("kind", [0, 1])
def test_polynomial_against_oracle(order, kind):
    r = np.random.default_rng(8)
    seen = set()
    for v in [10.0000001, 10.5, 12.0, 13.6, 14.001, 16.0, 16.001, 20.0, 28.0, 28.001, 50.0, 70.0, 70.001, 150.0, 230.0, 230.001,
              1e3, 1e5, 1e8] + list(np.exp(r.uniform(np.log(10.1), np.log(2000.0), 15))):
        # U_K of the tight dispatch: up to where mu_20 takes over, from the wide ranges' edges on
        lo = 1e-6 if v > 16 else (14.5 if v > 14 else 17.5 if v > 12 and kind == 0 else 19.5)
        hi = max(v * v / 3.24, 59.69) if v >= 13.6 else (30.0 if kind == 0 else 22.0 if v >= 12.5 else 20.0)
        x = np.concatenate([np.exp(r.uniform(np.log(lo), np.log(hi), 250)), lo + (hi - lo) * r.random(250) ** 4, [lo, hi]])
        x = np.ascontiguousarray(x[x < 1e8])
        f, cmax = np.empty_like(x), ctypes.c_double()
        K = order.poly(kind, 0, ctypes.c_double(v), *(a.ctypes.data_as(ctypes.c_void_p) for a in (x, f)),
                       ctypes.c_long(x.size), ctypes.byref(cmax))
        assert K == (4 if v > 230 else 6 if v > 70 else 9 if v > 28 else 13) and cmax.value < 0.25
        seen.add(K)
        vv = np.full_like(x, v)
        ref = (oracle.log_k if kind else oracle.log_i)(vv, x)
        err = oracle.rel_err(f, ref, oracle.error_scale("ik"[kind], vv, x))
        assert err.max() <= TOL, (v, x[err.argmax()], err.max())
    assert seen == {4, 6, 9, 13}


def test_polynomial_orders(order):
    """None up to order 10, past 1e150, or where several K serve one order."""
    x, f, c = np.array([25.0]), np.empty(1), ctypes.c_double()
    for v, mode, K in [(10.0, 0, 0), (9.0, 1, 0), (-20.0, 0, 0), (np.nan, 0, 0), (np.inf, 0, 0), (1e151, 0, 0), (20.0, 2, 0),
                       (20.0, 1, 13), (300.0, 1, 13), (300.0, 0, 4)]:
        assert order.poly(0, mode, ctypes.c_double(v), *(a.ctypes.data_as(ctypes.c_void_p) for a in (x, f)),
                          ctypes.c_long(1), ctypes.byref(c)) == K, (v, mode)
