"""Calls with one order for all arguments from 2^17 pairs on, where a block
computes the order's constants once: log I and log K against the oracle on a
sample, over the orders at which mu_20's scale or form changes, with x next to
30, on both sides of v^2 = 3.24 x and over every region.

Tolerance, in units of the error metric: from x = 18.4 on (expansions only)
truncation 3.1e-16, sums and logarithms 3e-16, roundings 2.2e-16: 1e-15;
below it the library's gate, 4e-15."""
import numpy as np
import pytest
import torch

import oracle
import paper_2409_08729_gb300 as lb

pytestmark = pytest.mark.gpu
ORDERS = [0.0, 0.3, 2.5, 8.0, 9.4, 10.0, 10.001, 10.9, 11.0, 12.0, 12.6964, 13.3, 13.59, 13.6, 14.5, 15.0, 15.39, 16.0,
          17.0, 20.0, 24.0, 28.0, 28.5, 70.0, 70.5, 100.0, 230.5, 1e4]


def _arguments(v, rng):
    """1000 arguments to check."""
    e = max(v * v / 3.24, 59.6925)
    return np.concatenate([rng.uniform(18.4, 32.0, 200), 30.0 + rng.uniform(-0.05, 0.15, 200),
                           e * (1.0 + rng.uniform(-1e-5, 1e-5, 100)), e * rng.uniform(1.0, 1.3, 200),
                           rng.uniform(30.0, 100.0, 100), np.exp(rng.uniform(np.log(1e-3), np.log(1e5), 200))])


@pytest.mark.parametrize("n", [(1 << 17) + 1, (1 << 20) + 1])
@pytest.mark.parametrize("kind", ["i", "k"])
def test_one_order_against_oracle(cuda, kind, n):
    fn = lb.log_i if kind == "i" else lb.log_k
    ref_fn = oracle.log_i if kind == "i" else oracle.log_k
    for v in ORDERS:
        rng = np.random.default_rng(int(100 * v) + n % 7)
        x = np.exp(rng.uniform(np.log(1e-3), np.log(1e4), n))
        at = rng.permutation(n)[:1000]
        x[at] = _arguments(v, rng)
        got = fn(v, torch.tensor(x, device=cuda)).cpu().numpy()[at]
        vv, xs = np.full(at.size, v), x[at]
        ref = ref_fn(vv, xs)
        err = oracle.rel_err(got, ref, oracle.error_scale(kind, vv, xs))
        over = err > np.where(xs >= 18.4, 1e-15, 4e-15)
        assert not over.any(), (v, xs[over][:3], err[over].max())


@pytest.mark.parametrize("n", [1 << 17, 1 << 20])
def test_the_blocks_constants_are_used(cuda, n):
    """The two forms of mu_20 round differently for a few pairs in a hundred:
    from these sizes on a call with one order is not the vector call's kernel."""
    x = torch.tensor(np.random.default_rng(5).uniform(30.0, 100.0, n), device=cuda)
    for fn in (lb.log_i, lb.log_k):
        a, b = fn(8.0, x), fn(torch.full_like(x, 8.0), x)
        assert not torch.equal(a, b) and float(((a - b).abs() / b.abs()).max()) <= 4e-15
