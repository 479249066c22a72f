"""The K integral by the trapezoid rule (csrc/lb_ktrap.cuh): its host build
against the oracle over every class, and the kernel at the sizes and class
mixes where its windows and chunks have edges.

Tolerances, in the units of the error metric.  Values: the result adds
-(a + b), v log(2a/x) and a logarithm, each with one or two roundings of at
most 2^-53 of the scale (3.3e-16 to 6.7e-16 in all), the rule's own error
(1.2e-16) and the fixed-point sum's (1e-16): 1e-15.  Derivatives (relative):
a quotient of two sums, six roundings, and the same two errors: 1.2e-15."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_08729_gb300", "csrc")
TOL, TOL_DX = 1e-15, 1.2e-15
SRC = r'''
#include "lb_ktrap.cuh"
extern "C" void kt(const double* v, const double* x, double* o, int* c, long n, int dx) {
  for (long i = 0; i < n; ++i) {
    c[i] = lb::kt_class(v[i], x[i], dx != 0);
    o[i] = dx ? lb::kt_eval<true>(v[i], x[i], c[i], lb_kt_exp2) : lb::kt_eval<false>(v[i], x[i], c[i], lb_kt_exp2);
  }
}
extern "C" int kt_band(double v, double x, int cls) { return lb::kt_band(v, x, cls); }
'''


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("ktrap")
    src, so = str(d / "kt.cpp"), str(d / "kt.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-o", so, src],
                   check=True)
    L = ctypes.CDLL(so)
    L.kt_band.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.c_int]

    def run(v, x, dx=False):
        v, x = np.ascontiguousarray(v, dtype=float), np.ascontiguousarray(x, dtype=float)
        o, c = np.empty_like(x), np.empty(x.size, dtype=np.int32)
        L.kt(*(a.ctypes.data_as(ctypes.c_void_p) for a in (v, x, o, c)), ctypes.c_long(x.size), int(dx))
        return o, c
    run.band = L.kt_band
    return run


def _pairs(n, seed, xmin=1e-300):
    """The fallback region of both dispatches (v <= 16, x <= 30, r <= 30),
    both sides of every class edge, integers and halves."""
    r = np.random.default_rng(seed)
    v = np.concatenate([r.uniform(0, 16, n), np.exp(r.uniform(np.log(1e-8), np.log(16), n)),
                        r.choice([0.0, 0.5, 1.0, 1.5, 2.0, 2.5, 7.5, 8.0, 16.0], n)])
    x = np.concatenate([np.exp(r.uniform(np.log(1e-3), np.log(30), 2 * n)), np.exp(r.uniform(np.log(xmin), 0, n))])
    r.shuffle(x)
    ve = r.uniform(0, 16, 4 * n)
    edge = np.select([np.arange(4 * n) % 4 == k for k in range(4)],
                     [np.full(4 * n, 2.0 ** -9), 4.5 - 1.5 * ve ** 2, 17.8 - 0.28 * ve ** 2, 31.0 - 0.09 * ve ** 2])
    ve, edge = ve[edge > 0], edge[edge > 0] * (1 + r.choice([-1e-6, 1e-6], int((edge > 0).sum())))
    v, x = np.concatenate([v, ve]), np.concatenate([x, edge])
    k = (x <= 30) & (v * v + x * x <= 900)
    return v[k], x[k]


@pytest.mark.parametrize("dx", [False, True])
def test_host_build_against_oracle(host, dx):
    v, x = _pairs(4000, 3 + dx)
    got, cls = host(v, x, dx)
    assert set(cls) == {1, 2, 3, 4, 5}
    if dx:
        ref = oracle.dlog_k_dx(v, x)
        err = np.abs(got - ref) / np.abs(ref)
    else:
        err = oracle.rel_err(got, oracle.log_k(v, x), oracle.error_scale("k", v, x))
    for c in range(1, 6):
        s = cls == c
        i = np.flatnonzero(s)[np.argmax(err[s])]
        assert err[i] <= (TOL_DX if dx else TOL), (c, err[i], v[i], x[i])


def test_any_pair(host):
    """Class 0 (a forced evaluation outside the other classes): large orders
    and arguments, against the oracle."""
    v = np.array([16.6, 40.0, 100.0, 1e3, 1e5, 3.0, 0.0, 20.0, 16.0])
    x = np.array([1e-6, 1e-3, 150.0, 2e3, 1.0, 2e3, 1e6, 1e-2, 40.0])
    got, cls = host(v, x)
    assert np.all(cls == 0)
    assert oracle.rel_err(got, oracle.log_k(v, x), oracle.error_scale("k", v, x)).max() <= TOL


def test_bands(host):
    """Every band is one of the eight that a queue entry has room for."""
    v, x = _pairs(300, 9)
    _, cls = host(v, x)
    b = [host.band(a, c, int(k)) for a, c, k in zip(v, x, cls)]
    assert min(b) >= 0 and max(b) <= 7
    assert host.band(16.0, 1e-3, 2) <= 7 and host.band(0.0, 4.0, 1) >= 0 and host.band(16.5, 1e-300, 2) <= 7


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 31, 33, 255, 257, 2047, 2049, 40001])
@pytest.mark.parametrize("dx", [False, True])
def test_kernel_windows(cuda, n, dx):
    """Every pair in the integral, all classes in one call, sizes around the
    chunk, block and window edges; one order per pair and one for all."""
    import torch
    import paper_2409_08729_gb300 as lb
    v, x = _pairs(8000, n + dx)
    keep = np.random.default_rng(n).permutation(v.size)[:n]
    v, x = v[keep], x[keep]
    tx = torch.tensor(x, device=cuda)
    for one in (False, True):
        vv = np.full_like(x, v[0]) if one else v
        ok = vv * vv + x * x <= 900
        tv = float(v[0]) if one else torch.tensor(v, device=cuda)
        got = (lb.log_k_dx if dx else lb.log_k)(tv, tx).cpu().numpy()
        if dx:
            ref = oracle.dlog_k_dx(vv, x)
            err, tol = np.abs(got - ref) / np.abs(ref), 4e-15
        else:
            ref = oracle.log_k(vv, x)
            err, tol = oracle.rel_err(got, ref, oracle.error_scale("k", vv, x)), 4e-15
        assert np.all(err[ok] <= tol), (one, float(err[ok].max()))
