"""Leaf-first LRU eviction against the oracle where it takes different routes: whole last_use values
and part of one, stamps that need several histogram passes, more evictions than one round takes, a
last_use value with more blocks than shared memory orders, and stamps that increase down a chain
(evicted one block at a time)."""
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


def _run(P, I, calls, cap, every_call=False):
    """calls: (chains [(inst, blocks, parent)], last_use); evicts after the last (or after each), compares the
    contents."""
    every = np.unique(np.concatenate([c[1] for ch, _ in calls for c in ch]))
    model = dict(W.MODEL_DEFAULT)
    st = dict(b=np.zeros(I, np.int32), qr=np.zeros(I, np.int32), q=np.zeros(I, np.int64), S=np.zeros(I, np.int64),
              M_KV=np.full(I, 10 ** 7, np.int64), B_max=np.full(I, 8, np.int32))
    none = dict(inst=np.zeros(0, np.uint32), state=np.zeros(0, np.uint32), L=np.zeros(0, np.uint32),
                out=np.zeros(0, np.uint32), rem=np.zeros(0, np.uint64))
    win = W.Window(chain_off=np.arange(every.size + 1, dtype=np.uint64), chain_hash=every,
                   prompt_tokens=np.full(every.size, 16, np.uint32), ttft_target=np.full(every.size, 1e6, np.float32),
                   tpot_target=np.full(every.size, 50.0, np.float32), session=np.zeros(every.size, np.uint32),
                   out_tokens=np.zeros(every.size, np.uint32))
    orc = Oracle(I, model, track_lru=True)
    orc.set_state(**st)
    orc.set_capacity(np.full(I, cap, np.uint64))
    orc.load_requests(none)
    total = max(sum(len(c[1]) for ch, _ in calls for c in ch if c[0] == i) for i in range(I))
    with P.Scheduler(I, np.full(I, cap, np.uint64), every.size, every.size, model,
                     table_load_factor=min(0.9, cap / (1.3 * total + 64)), probe_mode=P.PS_PROBE_LINEAR, track_lru=True,
                     max_active_requests=4) as s:
        s.load_instances(**st)
        s.load_requests(none)
        for chains, stamp in calls:
            off = np.zeros(len(chains) + 1, np.uint64)
            off[1:] = np.cumsum([len(c[1]) for c in chains])
            args = (np.array([c[0] for c in chains], np.uint32), off, np.concatenate([c[1] for c in chains]),
                    np.array([c[2] for c in chains], np.uint64))
            try:
                s.insert_chains(*args, last_use=stamp)
            except P.PSError as e:
                assert e.status == P.PS_ERR_CAPACITY, str(e)
            orc.insert_chains(*args, last_use=stamp)
            if every_call:
                s.advance_window(20.0, 1000, evict=True)
                orc.advance(20.0, 1000)
                assert s.cached_blocks().tolist() == [orc.cached_blocks(i) for i in range(I)]
                assert np.array_equal(s.score_window(win, want=("hits",))["hits"], orc.score_rows(win)["hits"])
        for _ in range(2):  # the second advance finds nothing over capacity
            s.advance_window(20.0, 1000, evict=True)
            orc.advance(20.0, 1000)
            assert s.cached_blocks().tolist() == [orc.cached_blocks(i) for i in range(I)]
            assert np.array_equal(s.score_window(win, want=("hits",))["hits"], orc.score_rows(win)["hits"])


def _blocks(rng, n):
    return rng.integers(2, 2 ** 63, n, dtype=np.int64).astype(np.uint64)


def _chains(rng, I, n, length, branch=0.3):
    out, seen = [], [[] for _ in range(I)]
    for _ in range(n):
        i = int(rng.integers(0, I))
        b = _blocks(rng, int(rng.integers(1, length + 1)))
        parent = int(seen[i][int(rng.integers(0, len(seen[i])))]) if seen[i] and rng.random() < branch else 0
        out.append((i, b, parent))
        seen[i].extend(b.tolist())
    return out


@pytest.mark.parametrize("stamps", [(0,), (0, 1, 2), (7, 3, 9), (2047, 2048, 5000), (3, 2500, 5_000_000, 4_000_000_000),
                                    (4_294_967_295, 0)])
@pytest.mark.parametrize("cap", [40, 400, 1500])
def test_stamps_and_partial_values(P, stamps, cap):
    rng = np.random.default_rng(cap + len(stamps))
    _run(P, 3, [(_chains(rng, 3, 60, 60), s) for s in stamps], cap)


@pytest.mark.parametrize("n", [1, 2, 1023, 1025, 16383, 16384, 16385, 20000])
@pytest.mark.parametrize("shape", ["one_chain", "many_chains"])
def test_one_value_around_the_shared_memory_limit(P, n, shape):
    rng = np.random.default_rng(n)
    if shape == "one_chain":
        chains = [(0, _blocks(rng, n), 0)]
    else:
        chains = [(0, _blocks(rng, min(16, n - k)), 0) for k in range(0, n, 16)]
    _run(P, 1, [(chains, 5)], max(1, n - n // 3))


def test_more_evictions_than_a_round(P):
    rng = np.random.default_rng(3)
    _run(P, 2, [([(i, _blocks(rng, 4000), 0) for i in (0, 1, 1)], k) for k in range(8)], 3000)


def test_children_newer_than_their_parents(P):
    rng = np.random.default_rng(4)
    first = _chains(rng, 4, 80, 30)
    # instance 0: continuations with a newer stamp; instance 1: a newer child of an old block further up;
    # the others stay in order
    later = [(i, _blocks(rng, 20), int(b[-1 if i == 0 else 0])) for i, b, _ in first if i < 2]
    _run(P, 4, [(first, 1), (later, 6), (_chains(rng, 4, 40, 30), 3)], 500)


def test_more_instances_than_a_round(P):
    rng = np.random.default_rng(6)
    _run(P, 300, [(_chains(rng, 300, 1500, 8), k) for k in range(3)], 20)


@pytest.mark.parametrize("I", [1, 5, 40])
def test_small_and_large_excess_in_turn(P, I):
    """Excesses on both sides of the one up to which blocks go one by one (64, and half the number of instances
    over capacity more), in calls that follow one another in every order; some instances have none."""
    rng = np.random.default_rng(I)
    calls = [([(i, _blocks(rng, 300), 0) for i in range(I)], 0)]
    sizes = [1, 64, 65, 0, 300, 200, 3, 80, 81, 82, 2, 64, 85, 299]
    for k, n in enumerate(sizes):
        over = [(i, _blocks(rng, n if i % 3 else max(1, n // 2)), 0) for i in range(I) if n and (i % 7 or I < 7)]
        calls.append((over or [(0, _blocks(rng, 1), 0)], k + 1))
    _run(P, I, calls, 300, every_call=True)
