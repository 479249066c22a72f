"""x-derivatives at half-odd orders, whose large-argument sums end after
v - 1/2 terms, and at their neighbours, whose sums do not: against the oracle
(relative, the library's gate of 4e-15), alone and among other orders."""
import numpy as np
import pytest
import torch

import oracle
import paper_2409_08729_gb300 as lb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1500, 150001])
@pytest.mark.parametrize("kind", ["i", "k"])
def test_half_odd_orders(cuda, kind, n):
    fn, ref_fn = (lb.log_i_dx, oracle.dlog_i_dx) if kind == "i" else (lb.log_k_dx, oracle.dlog_k_dx)
    rng = np.random.default_rng(n)
    half = np.arange(0, 14) + 0.5
    near = np.concatenate([np.nextafter(half, 0), np.nextafter(half, 99), half * (1 + 1e-9), half * (1 - 1e-7), [1.0, 2.0, 7.0]])
    v = rng.choice(np.concatenate([half, near]), n)
    x = np.exp(rng.uniform(np.log(25.0), np.log(1e4), n))
    s = rng.permutation(n)[:1500]
    got = fn(torch.tensor(v, device=cuda), torch.tensor(x, device=cuda)).cpu().numpy()[s]
    assert np.max(np.abs(got / ref_fn(v[s], x[s]) - 1)) <= 4e-15
    for order in (0.5, 1.5, 12.5):                    # one order for all
        vv = np.full(s.size, order)
        got = fn(order, torch.tensor(x, device=cuda)).cpu().numpy()[s]
        assert np.max(np.abs(got / ref_fn(vv, x[s]) - 1)) <= 4e-15, order
    # order 1/2 in closed form: sqrt(2/(pi x)) sinh x and sqrt(pi/(2x)) exp(-x)
    want = (1.0 if kind == "i" else -1.0) - 0.5 / x[s]
    got = fn(0.5, torch.tensor(x, device=cuda)).cpu().numpy()[s]
    assert np.max(np.abs(got / want - 1)) <= 4e-15
