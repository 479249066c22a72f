"""The FP32 kernel of the tight mode (warp_pairs32): slice, block and list
edges, the edge r = 14 between the expansion and the listed pairs, pointers
that 16-byte loads do not fit, outputs in place, and orders or arguments
whose squares leave single precision.  Gate: 2e-6 of the error scale."""
import numpy as np
import pytest
import torch

import oracle
import paper_2409_08729_gb300 as lb

pytestmark = pytest.mark.gpu
TOL32 = 2e-6
WIDE = 152 * 6 * 256 + 129          # just above the size where lanes take four pairs


def _pairs(n, seed):
    """A third on both sides of r = 14 within 1e-6, a third listed (all sort
    keys: x to 1e-37, v to 16), the rest over the domain."""
    r = np.random.default_rng(seed)
    v = np.exp(r.uniform(np.log(1e-6), np.log(1e4), n))
    x = np.exp(r.uniform(np.log(1e-3), np.log(1e4), n))
    k = np.arange(n) % 3
    a = r.uniform(0, np.pi / 2, n)
    v = np.where(k == 0, 14 * np.sin(a) * (1 + 1e-6 * r.choice([-1, 1], n)), v)
    x = np.where(k == 0, np.maximum(14 * np.cos(a), 1e-6), x)
    v = np.where(k == 1, r.choice([0.0, 0.5, 1.0, 3.3, 7.9, 13.9, 16.0], n), v)
    x = np.where(k == 1, np.exp(r.uniform(np.log(1e-37), np.log(14.5), n)), x)
    return v.astype(np.float32), x.astype(np.float32)


def _check(kind, v, x, got):
    v, x = np.broadcast_to(v, x.shape).astype(np.float64), x.astype(np.float64)
    ref = oracle.log_i(v, x) if kind == "i" else oracle.log_k(v, x)
    err = oracle.rel_err(got.astype(np.float64), ref, oracle.error_scale(kind, v, x))
    i = int(np.argmax(err))
    assert err[i] <= TOL32, (err[i], v[i], x[i], got[i], ref[i])


@pytest.mark.parametrize("kind", ["i", "k"])
@pytest.mark.parametrize("n", [1, 31, 33, 255, 257, 4097, WIDE])
def test_sizes(cuda, kind, n):
    fn = lb.log_i if kind == "i" else lb.log_k
    v, x = _pairs(n, n)
    tv, tx = torch.tensor(v, device=cuda), torch.tensor(x, device=cuda)
    got = fn(tv, tx)
    s = np.unique(np.concatenate([np.random.default_rng(1).integers(0, n, min(n, 3000)), np.arange(max(0, n - 130), n)]))
    _check(kind, v[s], x[s], got.cpu().numpy()[s])
    # the same bits one pair per lane (pointers off 16 bytes), in place, and with the order as a scalar
    bx, bv = torch.empty(n + 1, device=cuda), torch.empty(n + 1, device=cuda)
    bx[1:], bv[1:] = tx, tv
    assert torch.equal(fn(bv[1:], bx[1:]), got)
    assert torch.equal(fn(tv, tx, out=tx), got)
    tx = torch.tensor(x, device=cuda)
    one = torch.full_like(tx, 3.25)
    assert torch.equal(fn(3.25, tx), fn(one, tx))


@pytest.mark.parametrize("kind", ["i", "k"])
def test_lists_of_one_kind(cuda, kind):
    """Every pair listed (lists flush and keep a remainder), and none."""
    fn = lb.log_i if kind == "i" else lb.log_k
    r = np.random.default_rng(5)
    n = 40000
    for lo, hi in ((1e-3, 9.0), (15.0, 200.0)):
        v, x = r.uniform(0, 10, n).astype(np.float32), r.uniform(lo, hi, n).astype(np.float32)
        got = fn(torch.tensor(v, device=cuda), torch.tensor(x, device=cuda)).cpu().numpy()
        s = r.integers(0, n, 4000)
        _check(kind, v[s], x[s], got[s])


def test_squares_out_of_range(cuda):
    """v or x above 1e18: log I_v(x) = x - log(2 pi x)/2 for x >> v^2, and
    log(x/2) v - lgamma(v + 1) for v >> x^2, to single precision."""
    x = torch.tensor([1e19, 3e30, 1.0, 5.0], device=cuda)
    v = torch.tensor([2.0, 0.0, 1e19, 4e25], device=cuda)
    i, k = lb.log_i(v, x).cpu().numpy(), lb.log_k(v, x).cpu().numpy()
    want = np.array([1e19, 3e30] + [b * np.log(0.5 * a) - b * (np.log(b) - 1) for a, b in ((1.0, 1e19), (5.0, 4e25))])
    assert np.allclose(i, want, rtol=2e-6) and np.allclose(k, -want, rtol=2e-6)
