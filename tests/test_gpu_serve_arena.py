"""Arena of served FP32 log K requests: their integrals are evaluated in the
tile items, so nothing but their buffers counts against it."""
import numpy as np
import pytest
import torch

import paper_2409_08729_gb300 as lb
from paper_2409_08729_gb300 import workloads as W
from paper_2409_08729_gb300.serve import Server

pytestmark = pytest.mark.gpu


def test_fp32_k_needs_no_queue(cuda):
    n = 341 * 256                          # 3 x 4 n bytes: 1023 KiB of the 1 MiB arena
    v, x = (a.astype(np.float32) for a in W.robust_pairs(n, seed=21, vmax=30.0, xmin=1e-3, xmax=40.0))
    tv, tx = torch.tensor(v, device=cuda), torch.tensor(x, device=cuda)
    want = lb.log_k(tv, tx)
    with Server(arena_bytes=1 << 20, max_slots=4) as srv:
        o = np.empty_like(x)
        srv.wait(srv.submit("k", v, x, o), timeout=60)
        assert np.array_equal(o, want.cpu().numpy())
        # on device buffers nothing at all, whatever the size; again in the slot just freed
        big_v, big_x = tv.repeat(5), tx.repeat(5)
        for _ in range(2):
            big_o = torch.empty_like(big_x)
            srv.wait(srv.submit_device("k", big_v, big_x, big_o), timeout=60)
            assert torch.equal(big_o, want.repeat(5))
        # FP64 log K keeps its queues: 24 n bytes, refused as before
        with pytest.raises(lb.LogBesselError):
            srv.submit_device("k", tv.double(), tx.double(), torch.empty_like(tx.double()))
        d = torch.empty(20000, dtype=torch.float64, device=cuda)
        srv.wait(srv.submit_device("k", tv[:20000].double(), tx[:20000].double(), d), timeout=60)
        ref = lb.log_k(tv[:20000].double(), tx[:20000].double())
        assert float(((d - ref).abs() / ref.abs().clamp(min=1.0)).max()) <= 4e-15
