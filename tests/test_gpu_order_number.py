"""Orders given as Python numbers: past single precision's range they round to
an infinity as a tensor made from the number does, and the call under autograd
takes the same order as the plain one, without a copy from the host."""
import pytest
import torch

import paper_2409_08729_gb300 as lb

pytestmark = pytest.mark.gpu
INF = float("inf")


@pytest.mark.parametrize("grad", [False, True])
@pytest.mark.parametrize("v", [1e39, 3.4028235e38, 3.4028236e38, 1e300, INF])
def test_order_past_single_precision(cuda, v, grad):
    x = torch.tensor([0.5, 2.0, 1e5], dtype=torch.float32, device=cuda, requires_grad=grad)
    order = torch.tensor(v, dtype=torch.float32)
    for fn, sign in ((lb.log_i, -1.0), (lb.log_k, 1.0)):
        got = fn(v, x).detach()
        assert torch.equal(got, fn(order.to(cuda), x.detach()))
        if torch.isinf(order):
            assert torch.equal(got, torch.full_like(got, sign * INF))


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_order_under_autograd(cuda, dtype):
    x = torch.linspace(0.5, 50.0, 300, dtype=dtype, device=cuda, requires_grad=True)
    for fn in (lb.log_i, lb.log_k):
        for v in (0, 2.5, -0.5 if fn is lb.log_k else 0.1):
            assert torch.equal(fn(v, x).detach(), fn(v, x.detach()))
    # a copy from pageable memory cannot be captured; a fill can
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        y = lb.log_k(2.5, x)
    g.replay()
    assert torch.equal(y.detach(), lb.log_k(2.5, x.detach()))
