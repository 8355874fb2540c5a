"""Bulk insertion against the oracle: which blocks are cached after calls that repeat blocks, share
prefixes, name parents that come later in the same call, and spread over many tiles; and, where parents
come first, through the evictions that follow, the parent links and last-use stamps it leaves."""
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


def _forest(rng, I, n_chains, max_len):
    """Random prefix forests: chains that start at a root or continue a block of another chain, some
    repeating a chain's blocks; parents first."""
    chains, blocks = [], [[] for _ in range(I)]
    for _ in range(n_chains):
        i = int(rng.integers(0, I))
        n = int(rng.integers(0, max_len + 1))
        new = rng.integers(2, 2 ** 63, n, dtype=np.int64).astype(np.uint64)
        parent = 0
        if blocks[i] and rng.random() < 0.6:
            parent = int(blocks[i][int(rng.integers(0, len(blocks[i])))])
        kind = rng.random()
        if chains and kind < 0.2:  # an earlier chain again, a part of it or with a longer end
            j, ch, par = chains[int(rng.integers(0, len(chains)))]
            cut = int(rng.integers(0, len(ch) + 1))
            i, new, parent = j, np.concatenate([ch[:cut], new[:n // 3]]), par
        chains.append((i, new, parent))
        blocks[i].extend(new.tolist())
    return chains


def _csr(chains):
    off = np.zeros(len(chains) + 1, np.uint64)
    off[1:] = np.cumsum([len(c[1]) for c in chains])
    return (np.array([c[0] for c in chains], np.uint32), off,
            np.concatenate([c[1] for c in chains]).astype(np.uint64) if chains else np.zeros(0, np.uint64),
            np.array([c[2] for c in chains], np.uint64))


@pytest.mark.parametrize("parents_first", [True, False])
@pytest.mark.parametrize("I,n_chains,max_len,lf", [(1, 40, 3, 0.5), (3, 300, 40, 0.95), (2, 2600, 5, 0.5),
                                                   (5, 60, 2000, 0.9), (40, 700, 64, 0.75)])
def test_blocks_links_and_stamps(P, I, n_chains, max_len, lf, parents_first):
    rng = np.random.default_rng(I * 1000 + max_len)
    forests = [_forest(rng, I, n_chains, max_len) for _ in range(2)]
    if not parents_first:
        forests = [[f[k] for k in rng.permutation(len(f))] for f in forests]
    calls = [_csr(f) for f in forests]
    every = np.unique(np.concatenate([c[2] for c in calls]))
    per = max(int(sum((c[1][1:] - c[1][:-1])[c[0] == i].sum() for c in calls)) for i in range(I))
    cap = np.full(I, max(8, per * 2 // 3), np.uint64)  # the evictions take about a third
    model = dict(W.MODEL_DEFAULT)
    orc = Oracle(I, model, track_lru=True)
    st = dict(b=np.zeros(I, np.int32), qr=np.zeros(I, np.int32), q=np.zeros(I, np.int64), S=np.zeros(I, np.int64),
              M_KV=np.full(I, 10 ** 7, np.int64), B_max=np.full(I, 8, np.int32))
    orc.set_state(**st)
    orc.set_capacity(cap)
    none = dict(inst=np.zeros(0, np.uint32), state=np.zeros(0, np.uint32), L=np.zeros(0, np.uint32),
                out=np.zeros(0, np.uint32), rem=np.zeros(0, np.uint64))
    win = W.Window(chain_off=np.arange(every.size + 1, dtype=np.uint64), chain_hash=every,  # one block a request
                   prompt_tokens=np.full(every.size, 16, np.uint32), ttft_target=np.full(every.size, 1e6, np.float32),
                   tpot_target=np.full(every.size, 50.0, np.float32), session=np.zeros(every.size, np.uint32),
                   out_tokens=np.zeros(every.size, np.uint32))
    with P.Scheduler(I, cap, every.size, every.size, model, table_load_factor=lf * 2 / 3, probe_mode=P.PS_PROBE_LINEAR,
                     track_lru=True, max_active_requests=4) as s:
        s.load_instances(**st)
        s.load_requests(none)
        orc.load_requests(none)
        for k, (inst, off, hashes, parent) in enumerate(calls):
            try:
                s.insert_chains(inst, off, hashes, parent, last_use=5 - 3 * k)  # the second call's stamps are older
            except P.PSError as e:
                assert e.status == P.PS_ERR_CAPACITY, str(e)  # above its capacity until the eviction
            orc.insert_chains(inst, off, hashes, parent, last_use=5 - 3 * k)
            assert s.cached_blocks().tolist() == [orc.cached_blocks(i) for i in range(I)]
            assert np.array_equal(s.score_window(win, want=("hits",))["hits"], orc.score_rows(win)["hits"])
            if not parents_first or (I > 1 and k == 0):
                continue  # (a child cached before its parent has no link to it)
            s.advance_window(20.0, 1000, evict=True)
            orc.advance(20.0, 1000)
            assert s.cached_blocks().tolist() == [orc.cached_blocks(i) for i in range(I)]
            assert np.array_equal(s.score_window(win, want=("hits",))["hits"], orc.score_rows(win)["hits"])
