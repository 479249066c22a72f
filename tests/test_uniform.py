"""The uniform expansions in fixed point (csrc/lb_uniform.cuh): the host build
against the oracle at the edges of each number of terms and of the range of
r; and the term counts of mu_20 (csrc/muterms_table.h).

Tolerances, in the units of the error metric.  Values: truncation at the
regions' edges 4e-16, the fixed-point logarithms (2^-53 each, times v) 2.2e-16,
two roundings of the result 2.2e-16: 1e-15.  Derivatives (relative): the
truncation counts K-fold near the edges, eight roundings: 2.5e-15."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_08729_gb300", "csrc")
TOL, TOL_DX = 1e-15, 2.5e-15
SRC = r'''
#include "lb_uniform.cuh"
#define LB_MUT_TABLE static const
#include "muterms_table.h"
extern "C" void uf(const double* v, const double* x, const int* cap, double* o, int* K, long n, int kind, int dx, int more) {
  for (long i = 0; i < n; ++i) {
    const double s = fma(v[i], v[i], x[i] * x[i]);
    K[i] = lb::uni_ok(s, x[i]) ? (dx ? lb::uni_terms_dx((float)s, cap[i]) : lb::uni_terms((float)s, cap[i])) : -1;
    if (K[i] < 0) continue;
    const int m = K[i] + more > 13 ? 13 : K[i] + more;
    o[i] = dx ? lb::u_dx_fx(kind, v[i], x[i], s, K[i], m) : lb::u_fx(kind, v[i], x[i], s, K[i], m);
  }
}
extern "C" void mut(const float* A, const float* w, int* o, long n) {
  for (long i = 0; i < n; ++i) {
    const int ia = (int)(lb::ix_fbits(A[i]) >> 22) - LB_MUT_A_BASE, iw = (int)(lb::ix_fbits(w[i]) >> 22) - LB_MUT_W_BASE;
    const int ca = ia < 0 ? 0 : (ia > LB_MUT_A_CELLS ? LB_MUT_A_CELLS : ia);
    const int cw = iw < 0 ? 0 : (iw > LB_MUT_W_CELLS ? LB_MUT_W_CELLS : iw);
    o[i] = lb_mut[cw * (LB_MUT_A_CELLS + 1) + ca];
  }
}
'''


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("uniform")
    src, so = str(d / "u.cpp"), str(d / "u.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-o", so, src],
                   check=True)
    return ctypes.CDLL(so)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _pairs(dx):
    """The U regions: log-uniform pairs, both sides of the order thresholds, of
    the half octaves of r^2 where the number of terms steps, and small x."""
    r = np.random.default_rng(11)
    v = np.concatenate([np.exp(r.uniform(np.log(16.001), np.log(1e5), 1500)), r.uniform(0.7, 16.0, 1000),
                        np.repeat([16.05, 28.0, 28.01, 70.0, 70.01, 230.0, 230.01], 100)])
    x = np.concatenate([np.exp(r.uniform(np.log(1e-6), np.log(1e5), 1500)), r.uniform(25.001, 59.0, 1000),
                        np.exp(r.uniform(np.log(1e-6), np.log(400.0), 700))])
    e = np.arange(18, 40)
    s = np.concatenate([768.0 * 2.0 ** ((e - 18) / 2.0), 512.0 * 2.0 ** ((e - 18) // 2), 768.0 * 2.0 ** ((e - 18) // 2)])
    s = np.concatenate([s * (1 - 1e-6), s * (1 + 1e-6)]) / (0.58 if dx else 1.0)
    c = r.uniform(0.0, 0.95, s.size)
    vv, xx = np.sqrt(s * (1 - c * c)), np.sqrt(s) * c
    ok = vv > 16.0
    v, x = np.concatenate([v, vv[ok]]), np.concatenate([x, xx[ok]])
    ok = ~((x > 59.6925) & (v * v < 3.24 * x)) & ~((x > 30.0) & (v < 13.6))
    return np.ascontiguousarray(v[ok]), np.ascontiguousarray(x[ok])


@pytest.mark.parametrize("dx", [False, True])
@pytest.mark.parametrize("kind", [0, 1])
def test_fixed_point_expansions(host, kind, dx):
    v, x = _pairs(dx)
    cap = np.where(v > 230, 4, np.where(v > 70, 6, np.where(v > 28, 9, 13))).astype(np.int32)
    o, o2, K = np.empty_like(v), np.empty_like(v), np.empty(v.size, dtype=np.int32)
    host.uf(_p(v), _p(x), _p(cap), _p(o), _p(K), ctypes.c_long(v.size), kind, int(dx), 0)
    assert K.min() >= 4 and set(K) >= {4, 5, 6, 7, 8, 9, 13}
    host.uf(_p(v), _p(x), _p(cap), _p(o2), _p(K), ctypes.c_long(v.size), kind, int(dx), 3)
    assert np.array_equal(o, o2)                      # a pair's result does not depend on its warp's count
    if dx:
        ref = (oracle.dlog_k_dx if kind else oracle.dlog_i_dx)(v, x)
        err = np.abs(o / ref - 1)
    else:
        ref = (oracle.log_k if kind else oracle.log_i)(v, x)
        err = oracle.rel_err(o, ref, oracle.error_scale("ik"[kind], v, x))
    assert err.max() <= (TOL_DX if dx else TOL), (err.max(), v[err.argmax()], x[err.argmax()], K[err.argmax()])


def test_range_of_r(host):
    """Outside [16.04, 1e150], and for a subnormal x, the other form serves."""
    v = np.array([16.03, 16.05, 1e149, 2e150, 20.0, 20.0])
    x = np.array([1e-3, 1e-3, 1.0, 1.0, 1e-310, 3e-308])
    K, o = np.empty(6, dtype=np.int32), np.zeros(6)
    host.uf(_p(v), _p(x), _p(np.full(6, 4, dtype=np.int32)), _p(o), _p(K), ctypes.c_long(6), 0, 0, 0)
    assert list(K > 0) == [False, True, True, False, False, True]


def test_mu_term_counts(host):
    """n: the terms after the n-th are below 2^-56 (or n = 20); h: those from the
    h-th on below 1e-3; over both of mu_20's ranges (single-precision A, w)."""
    r = np.random.default_rng(12)
    x = np.exp(r.uniform(np.log(18.5), np.log(1e7), 20000))
    v = np.where(r.random(x.size) < 0.5, r.uniform(0, 13.6, x.size), r.random(x.size) * np.sqrt(3.24 * x))
    v = np.minimum(v, np.where(x > 59.6925, np.maximum(np.sqrt(3.24 * x), 13.6), np.where(x > 22, 13.6, 9.5)))
    w = (1.0 / (8.0 * x)).astype(np.float32)
    A = (4.0 * v * v / (8.0 * x)).astype(np.float32)
    o = np.empty(x.size, dtype=np.int32)
    host.mut(_p(A), _p(w), _p(o), ctypes.c_long(x.size))
    n, h = o & 255, o >> 8
    assert n.min() >= 1 and n.max() <= 20 and h.max() <= 20
    t = np.ones(x.size)
    for k in range(1, 21):
        t *= np.abs(A.astype(float) - (2 * k - 1) ** 2 * w.astype(float)) / k
        assert np.all(t[k > n] < 1.5e-17) and np.all(t[k >= h + 1] < 1.1e-3), k
