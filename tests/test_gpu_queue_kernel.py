"""The K integral's own kernel, which serves calls from 2^17 pairs on: few and
many pairs of a call in the integral, around the edges of its chunks, blocks
and windows, against the oracle; and the vMF log-normaliser's orders up to 16
from 2^17 values on, which take the one-order kernel.

Gates: the library's 4e-15 (values in the error metric, derivatives relative)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2409_08729_gb300 as lb
from paper_2409_08729_gb300 import _binding as B
from paper_2409_08729_gb300 import vmf

pytestmark = pytest.mark.gpu
TOL = 4e-15


def _integral_pairs(m, rng):
    """Pairs in the K integral of values and derivatives, every class but the general one."""
    v = np.where(rng.random(m) < 0.3, rng.choice([0.0, 0.5, 1.0, 2.0, 2.5, 8.0, 16.0], m), rng.uniform(0.0, 16.0, m))
    x = np.where(rng.random(m) < 0.3, np.exp(rng.uniform(np.log(1e-300), np.log(1e-2), m)), rng.uniform(1e-2, 13.9, m))
    return v, x


@pytest.mark.parametrize("dx", [False, True])
@pytest.mark.parametrize("m", [0, 1, 31, 33, 2047, 40001, 131072])
def test_pairs_in_the_queue(cuda, m, dx):
    n = (1 << 17) + 5
    m = n if m == 131072 else m                        # every pair of the call
    rng = np.random.default_rng(m + dx)
    v, x = rng.uniform(0.0, 300.0, n), rng.uniform(60.0, 300.0, n)       # expansions only
    at = rng.permutation(n)[:m]
    v[at], x[at] = _integral_pairs(m, rng)
    fn, ref_fn = (lb.log_k_dx, oracle.dlog_k_dx) if dx else (lb.log_k, oracle.log_k)
    before = B.profile_read()["lb_kint_kernel"][0]
    got = fn(torch.tensor(v, device=cuda), torch.tensor(x, device=cuda)).cpu().numpy()
    assert B.profile_read()["lb_kint_kernel"][0] == before + 1           # the queue's kernel ran
    s = np.unique(np.concatenate([at[:6000], rng.integers(0, n, 300)]))
    ref = ref_fn(v[s], x[s])
    err = np.abs(got[s] / ref - 1) if dx else oracle.rel_err(got[s], ref, oracle.error_scale("k", v[s], x[s]))
    assert err.max() <= TOL, (err.max(), v[s][err.argmax()], x[s][err.argmax()])


@pytest.mark.parametrize("order", [0.0, 0.5, 2.5, 9.75, 16.0])
def test_one_order_in_the_queue(cuda, order):
    n = (1 << 20) + 7
    rng = np.random.default_rng(int(8 * order))
    x = np.exp(rng.uniform(np.log(1e-4), np.log(60.0), n))
    got = lb.log_k(order, torch.tensor(x, device=cuda)).cpu().numpy()
    s = rng.integers(0, n, 4000)
    vv = np.full(s.size, order)
    err = oracle.rel_err(got[s], oracle.log_k(vv, x[s]), oracle.error_scale("k", vv, x[s]))
    assert err.max() <= TOL, (err.max(), x[s][err.argmax()])


@pytest.mark.parametrize("d", [2, 3, 22, 27, 28, 29, 30, 31, 32, 33, 34, 36])
def test_vmf_orders_from_2_17_values_on(cuda, d):
    n = 1 << 17
    rng = np.random.default_rng(d)
    x = np.exp(rng.uniform(np.log(1e-3), np.log(2e3), n))
    at = rng.permutation(n)[:2000]
    x[at[:1000]] = rng.uniform(29.5, 32.0, 1000)
    nu = 0.5 * d - 1.0
    e = max(nu * nu / 3.24, 59.6925)
    x[at[1000:1400]] = e * (1.0 + rng.uniform(-1e-3, 0.1, 400))
    got = vmf.log_c(d, torch.tensor(x, device=cuda)).cpu().numpy()[at]
    xs, vv = x[at], np.full(at.size, nu)
    li = oracle.log_i(vv, xs)
    want = nu * np.log(xs) - 0.5 * d * np.log(2 * np.pi) - li
    # each of the three terms correct to 1e-15 of its size (the error of log I), and the sum's roundings
    scale = np.abs(nu * np.log(xs)) + 0.5 * d * np.log(2 * np.pi) + np.maximum(np.abs(li), oracle.error_scale("i", vv, xs))
    assert np.max(np.abs(got - want) / scale) <= 1e-15
