"""FP32 calls at arguments down to the subnormals, orders on both sides of 14
(the merged expansion's edge) and far above: against the oracle, at the
FP32-mixed gate of 2e-6 of the error scale."""
import numpy as np
import pytest
import torch

import oracle
import paper_2409_08729_gb300 as lb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 300001])       # one pair per lane, four per lane
@pytest.mark.parametrize("kind", ["i", "k"])
def test_tiny_arguments(cuda, kind, n):
    v = np.array([0.5, 5.0, 13.9, 14.0, 14.1, 14.5, 15.39, 15.9, 16.0, 16.5, 70.0, 1e3, 1e5, 1e8, 1e12])
    x = np.array([4e-45, 1e-44, 1e-40, 1e-38, 1.2e-38, 1e-36, 1e-30, 1e-25, 5.4e-20, 5.5e-20, 1e-15, 1e-6])
    v, x = (a.ravel().astype(np.float32) for a in np.meshgrid(v, x))
    reps = -(-n // v.size)
    tv, tx = torch.tensor(v, device=cuda).repeat(reps), torch.tensor(x, device=cuda).repeat(reps)
    got = (lb.log_i if kind == "i" else lb.log_k)(tv, tx).view(reps, -1)
    assert torch.equal(got[0], got[-1])
    got, v, x = got[0].double().cpu().numpy(), v.astype(float), x.astype(float)
    ref = (oracle.log_i if kind == "i" else oracle.log_k)(v, x)
    err = oracle.rel_err(got, ref, oracle.error_scale(kind, v, x))
    assert err.max() <= 2e-6, (err.max(), v[err.argmax()], x[err.argmax()])
