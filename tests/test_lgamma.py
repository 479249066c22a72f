"""lgamma(v + 1) in integers (csrc/lb_lgamma.cuh): the host build against
40-digit values at the pieces' edges and between.  Tolerance: 5e-17 absolute
(coefficients and truncations 2^-56) and the result's rounding, 2^-53."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_08729_gb300", "csrc")
SRC = r'''
#include "lb_lgamma.cuh"
extern "C" void lg(const double* v, double* o, int* ok, long n) {
  for (long i = 0; i < n; ++i) { ok[i] = lb::lg_ok(v[i]); o[i] = ok[i] ? lb::lg_lgamma1p(v[i]) : 0.0; }
}
'''


def test_lgamma1p(tmp_path):
    mpmath = pytest.importorskip("mpmath")
    src, so = str(tmp_path / "l.cpp"), str(tmp_path / "l.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-o", so, src],
                   check=True)
    L = ctypes.CDLL(so)
    edges = np.concatenate([2.0 ** e * (1 + np.arange(8) / 8) for e in range(5)]) - 1.0
    edges = edges[edges < 17.0]
    v = np.concatenate([edges, np.nextafter(edges[1:], 0), np.nextafter(edges, 99), [5e-324, 1e-300, 1e-17, 1e-9],
                        np.random.default_rng(3).uniform(0, 17, 3000), [np.nextafter(17.0, 0)]])
    o, ok = np.empty_like(v), np.empty(v.size, dtype=np.int32)
    L.lg(*(a.ctypes.data_as(ctypes.c_void_p) for a in (v, o, ok)), ctypes.c_long(v.size))
    assert ok.all() and o[0] == 0.0                        # lgamma(1)
    with mpmath.workdps(40):
        for vi, oi in zip(v, o):
            ref = mpmath.loggamma(mpmath.mpf(float(vi)) + 1)
            assert abs(oi - ref) <= 5e-17 + abs(ref) * 2.0 ** -53, vi
    bad = np.array([17.0, 1e300, np.inf, np.nan, -1e-9, -0.5])
    L.lg(*(a.ctypes.data_as(ctypes.c_void_p) for a in (bad, o, ok)), ctypes.c_long(bad.size))
    assert not ok[:6].any()
