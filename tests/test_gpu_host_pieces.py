"""Host-buffer calls at sizes where the last pieces are cut differently (what
remains is below one chunk, between one and two, or a scrap): the bits of the
same call in another chunk size, every result written."""
import numpy as np
import pytest

import paper_2409_08729_gb300 as lb
from paper_2409_08729_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("chunks", [0.4, 1.0, 1.9, 2.0, 2.876, 3.87, 3.9, 5.1])
def test_last_pieces(cuda, dtype, chunks):
    chunk = 131072
    for n in (int(chunk * chunks), int(chunk * chunks) + 1):
        v, x = (a.astype(dtype) for a in W.robust_pairs(n, seed=n % 89, vmax=1e3, xmin=1e-3, xmax=1e3))
        for fn in ("log_i", "log_k"):
            out = np.full_like(x, 12345.0)
            lb.host_eval(fn, v, x, out=out, chunk=chunk)
            assert np.array_equal(out, lb.host_eval(fn, v, x, chunk=1 << 22), equal_nan=True), (fn, n)
