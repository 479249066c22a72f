"""FP64 calls take one of four kernels by their size: both sides of every
edge, values and derivatives, mixed and single orders, against the oracle on a
sample (the last pairs among it), at the gates of the parity tests."""
import numpy as np
import pytest
import torch

import oracle
import paper_2409_08729_gb300 as lb
from paper_2409_08729_gb300 import vmf
from paper_2409_08729_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 4e-15


@pytest.mark.parametrize("kind", ["i", "k"])
@pytest.mark.parametrize("n", [2, 63, 65, 2000, 2001, (1 << 17) - 1, 1 << 17, (1 << 20) - 1, 1 << 20])
def test_both_sides_of_every_route(cuda, kind, n):
    v, x = W.robust_pairs(n, seed=n % 1009, vmax=300.0, xmin=1e-3, xmax=300.0)
    s = np.unique(np.concatenate([np.random.default_rng(2).integers(0, n, 600), np.arange(max(0, n - 70), n)]))
    tx = torch.tensor(x, device=cuda)
    for order in (None, 4.25):
        vv = np.full(s.size, order) if order else v[s]
        tv = order if order else torch.tensor(v, device=cuda)
        ref = oracle.log_i(vv, x[s]) if kind == "i" else oracle.log_k(vv, x[s])
        got = (lb.log_i if kind == "i" else lb.log_k)(tv, tx).cpu().numpy()[s]
        err = oracle.rel_err(got, ref, oracle.error_scale(kind, vv, x[s]))
        assert err.max() <= TOL, (order, err.max(), vv[err.argmax()], x[s][err.argmax()])
        ref = oracle.dlog_i_dx(vv, x[s]) if kind == "i" else oracle.dlog_k_dx(vv, x[s])
        got = (lb.log_i_dx if kind == "i" else lb.log_k_dx)(tv, tx).cpu().numpy()[s]
        assert np.max(np.abs(got / ref - 1)) <= TOL, order


@pytest.mark.parametrize("n", [1, 2000, 2001, 300000])
def test_vmf_routes(cuda, n):
    """log C_d and its derivative stored by the tile kernels: against
    log I and d/dx log I of the same concentrations, and the limits."""
    d = 2048
    k = torch.tensor(np.exp(np.random.default_rng(n).uniform(np.log(20.0), np.log(20000.0), n)), device=cuda)
    nu = 0.5 * d - 1.0
    want = nu * torch.log(k) - 0.5 * d * np.log(2 * np.pi) - lb.log_i(nu, k)
    got = vmf.log_c(d, k)
    assert float(((got - want).abs() / (nu * torch.log(k))).max()) <= TOL
    dd, ratio = vmf.log_c(d, k, deriv=True), lb.log_i_dx(nu, k)
    assert float(((dd - (nu / k - ratio)).abs() / ratio).max()) <= TOL
    e = vmf.log_c(d, torch.tensor([0.0, -1.0, float("nan")], dtype=torch.float64, device=cuda)).cpu().numpy()
    lim = float(torch.lgamma(torch.tensor(d / 2.0, dtype=torch.float64))) - np.log(2) - 0.5 * d * np.log(np.pi)
    assert abs(e[0] - lim) <= TOL * abs(lim) and np.isnan(e[1]) and np.isnan(e[2])
    e = vmf.log_c(d, torch.tensor([0.0, float("inf")], dtype=torch.float64, device=cuda), deriv=True).cpu().numpy()
    assert e[0] == 0.0 and e[1] == -1.0


@pytest.mark.parametrize("d", [2, 3, 33, 34, 35, 300])
def test_vmf_order_in_either_kernel(cuda, d):
    """Orders d/2 - 1 up to 16 take the one-order kernel, larger ones the
    general kernel: log C_d of both against the oracle, over each expansion."""
    x = np.concatenate([np.geomspace(1e-3, 2e3, 2400), [18.49, 18.5, 18.51, 58.9, 59.0]])
    nu = 0.5 * d - 1.0
    li = oracle.log_i(np.full(x.size, nu), x)
    want = nu * np.log(x) - 0.5 * d * np.log(2 * np.pi) - li
    got = vmf.log_c(d, torch.tensor(x, device=cuda)).cpu().numpy()
    # each of the three terms correct to TOL of its size, and the roundings of the sum
    scale = np.abs(nu * np.log(x)) + 0.5 * d * np.log(2 * np.pi) + np.maximum(
        np.abs(li), oracle.error_scale("i", np.full(x.size, nu), x))
    assert np.max(np.abs(got - want) / scale) <= TOL
