"""Scoring at the row widths where its block changes size: 257 .. 512 instances take 128 threads, up to
1024 take 256; rows that are not a multiple of 4 wide go by single words.  Every output must equal the
oracle's, bit for bit."""
import numpy as np
import pytest

import workload as W
from oracle import Oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("a CUDA device is required for the gpu tests")
    import paper_2609_33224_gb300 as P
    P.build()
    return P


@pytest.mark.parametrize("R", [1, 700])  # 700 rows: blocks take an odd or an even number of rows
@pytest.mark.parametrize("I", [256, 257, 260, 509, 512, 513, 516, 1024, 1025])
def test_row_widths(P, I, R):
    wl = W.generate(0, seed=5, num_instances=I, window_requests=R, num_sessions=max(4, R // 6), cap_blocks=1024, b_hi=8,
                    b_max=64)
    o = Oracle(I, wl.model).load(wl.instances).score_rows(wl.window)
    with P.Scheduler(I, wl.instances.cap_blocks, R, int(wl.window.chain_off[-1]), wl.model, table_load_factor=0.5) as s:
        s.load_workload_instances(wl.instances)
        g = s.score_window(wl.window)
    for k in ("hits", "tpot", "ttft", "cls", "best", "path"):
        a, b = np.ascontiguousarray(g[k]), np.ascontiguousarray(o[k])
        assert a.dtype.itemsize == b.dtype.itemsize and a.tobytes() == b.tobytes(), k
