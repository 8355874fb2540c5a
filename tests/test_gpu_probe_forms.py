"""Hit lengths where the probe changes form: few pairs (a warp each) and many (a lane each, buckets read
by quads), instance counts that are not whole quads or chunks, rows derived from a base that most
instances cache in full (searched a lane each), and windows around the size up to which every earlier
request is compared directly."""
import numpy as np
import pytest

import workload as W
from oracle import Oracle
from tests.helpers import make_window

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("a CUDA device is required for the gpu tests")
    import paper_2609_33224_gb300 as P
    P.build()
    return P


def _check(P, ins, win, lf):
    orc = Oracle(ins.I, W.MODEL_DEFAULT).load(ins)
    with P.Scheduler(ins.I, ins.cap_blocks, win.R, int(win.chain_off[-1]), W.MODEL_DEFAULT, table_load_factor=lf) as s:
        s.load_workload_instances(ins)
        g, o = s.score_window(win), orc.score_rows(win)
        for k in ("hits", "cls", "best", "path"):
            assert np.array_equal(g[k], o[k]), k
        d, e = s.schedule_window(win), orc.schedule(win)
        for k in ("assign", "path", "hit_chosen"):
            assert np.array_equal(d[k], e[k]), k


@pytest.mark.parametrize("I", [3, 63, 64, 65, 127, 254, 255, 256, 257, 1021])
@pytest.mark.parametrize("R", [1, 2, 32, 33, 34, 200])
def test_instances_and_window_sizes(P, I, R):
    wl = W.generate(0, seed=I + R, num_instances=I, window_requests=R, num_sessions=max(4, R // 2), cap_blocks=1500,
                    fill_lo=0.9, fill_hi=1.0)
    _check(P, wl.instances, wl.window, 0.93)


@pytest.mark.parametrize("I", [9, 300])
def test_base_cached_everywhere(P, I):
    """A request that is the bare system prompt, cached in full on every instance, is a prefix of all later
    ones; some instances also cache parts of the sessions."""
    rng = np.random.default_rng(I)
    sys = rng.integers(0, 1 << 17, 16 * 40).astype(np.uint32)
    sess = [np.concatenate([sys, rng.integers(0, 1 << 17, 16 * 200).astype(np.uint32)]) for _ in range(6)]
    reqs = [(sys, 2000.0, 50.0)]
    for k in range(90):
        t = sess[int(rng.integers(0, 6))]
        reqs.append((t[:16 * 40 + int(rng.integers(1, 16 * 200))], 2000.0, 50.0))
    chains, inst = [], []
    for i in range(I):
        chains.append(W.chain_from_tokens(sys))
        inst.append(i)
        if i % 3 == 0:
            t = sess[i % 6]
            chains.append(W.chain_from_tokens(t[:16 * int(rng.integers(41, 240))]))
            inst.append(i)
    off = np.zeros(len(chains) + 1, np.uint64)
    off[1:] = np.cumsum([c.size for c in chains])
    ins = W.Instances(b=np.ones(I, np.int32), qr=np.zeros(I, np.int32), q=rng.integers(0, 5000, I).astype(np.int64),
                      S=np.zeros(I, np.int64), M_KV=np.full(I, 10 ** 7, np.int64), B_max=np.full(I, 64, np.int32),
                      cap_blocks=np.full(I, 2000, np.uint64), chain_inst=np.array(inst, np.uint32), chain_off=off,
                      chain_hash=np.concatenate(chains).astype(np.uint64), chain_parent=np.zeros(len(chains), np.uint64))
    _check(P, ins, make_window(reqs), 0.5)
