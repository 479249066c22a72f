"""Calls on both sides of where log I's derivative and the paper's dispatches
change their tiles: against the same pairs in calls of fewer than 2^17, which
take another kernel."""
import pytest
import torch

import paper_2409_08729_gb300 as lb
from paper_2409_08729_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("edge", ["low", "high"])
def test_both_sides(cuda, edge):
    sms = torch.cuda.get_device_properties(cuda).multi_processor_count
    at = sms * 6 * 512 // 4 * 5 if edge == "low" else sms * 3 * 2048
    v, x = W.robust_pairs(at + 1, seed=3, vmax=300.0, xmin=1e-2, xmax=300.0)
    v, x = torch.tensor(v, device=cuda), torch.tensor(x, device=cuda)
    for name, mode in (("log_i_dx", "tight"), ("log_i", "paper_gpu"), ("log_i_dx", "paper_cpu_order")):
        fn = getattr(lb, name)
        want = torch.cat([fn(v[i:i + 100000], x[i:i + 100000], mode=mode) for i in range(0, at + 1, 100000)])
        for n in (at, at + 1):
            got = fn(v[:n], x[:n], mode=mode)
            err = (got - want[:n]).abs() / want[:n].abs().clamp(min=1.0 if name == "log_i" else 0.0)
            assert float(err.max()) <= 4e-15, (name, mode, n)
