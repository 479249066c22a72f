"""Results written over the arguments (out is x, as the header allows) or over
the orders (out is v, which the kernels read before they write too): the bits
of a call with a buffer of its own, in every route."""
import pytest
import torch

import paper_2409_08729_gb300 as lb
from paper_2409_08729_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 1999, 40001, 300001, (1 << 20) + 3])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_in_place(cuda, dtype, n):
    v, x = W.robust_pairs(n, seed=n % 97, vmax=200.0, xmin=1e-3, xmax=200.0)
    v, x = torch.tensor(v, device=cuda).to(dtype), torch.tensor(x, device=cuda).to(dtype)
    names = ["log_i", "log_k"] + (["log_i_dx", "log_k_dx"] if dtype == torch.float64 else [])
    for name in names:
        fn = getattr(lb, name)
        want = fn(v, x)
        a, b = x.clone(), v.clone()
        fn(v, a, out=a)
        fn(b, x, out=b)
        for got in (a, b):
            assert bool(((got == want) | ((got - want).abs() <= 1e-15 * want.abs().clamp(min=1.0))).all()), name
