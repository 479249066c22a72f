"""Calls of up to 2000 FP64 pairs, a warp per pair: neighbours of other regions
and domain edges in a block change nothing, so each pair's result in a mixed
call has the bits of a call with that pair alone."""
import numpy as np
import pytest
import torch

import paper_2409_08729_gb300 as lb
from paper_2409_08729_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["log_i", "log_k", "log_i_dx", "log_k_dx"])
def test_mixed_call_equals_single_pairs(cuda, name):
    fn = getattr(lb, name)
    v, x = W.robust_pairs(180, seed=17, vmax=400.0, xmin=1e-4, xmax=400.0)
    ev, ex = W.edge_pairs()
    p = np.random.default_rng(3).permutation(180 + ev.size)
    tv = torch.tensor(np.concatenate([v, ev])[p], device=cuda)
    tx = torch.tensor(np.concatenate([x, ex])[p], device=cuda)
    whole = fn(tv, tx)
    alone = torch.cat([fn(tv[i:i + 1], tx[i:i + 1]) for i in range(tx.numel())])
    same = (whole == alone) | (torch.isnan(whole) & torch.isnan(alone))
    assert bool(same.all()), (tv[~same][:3], tx[~same][:3])
    # the last warps of a block past the end of a call write nothing
    out = torch.full_like(tx, 7.0)
    fn(tv[:63], tx[:63], out=out[:63])
    assert bool((out[63:] == 7.0).all())
