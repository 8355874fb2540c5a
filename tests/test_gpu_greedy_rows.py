"""The greedy pass where its deciding block changes shape: instance counts around its warp and
instances-per-thread boundaries, windows around the probe lag, equal keys, and states that need
64-bit sums.  Every decision and the pending state must equal the oracle's."""
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


def _check(P, model, ins, win, mode=1):
    orc = Oracle(ins.I, model).load(ins)
    with P.Scheduler(ins.I, ins.cap_blocks, win.R, int(win.chain_off[-1]), model, table_load_factor=0.5,
                     probe_mode=mode) as s:
        s.load_workload_instances(ins)
        g = s.schedule_window(win)
        o = orc.schedule(win)
        for k in ("assign", "path", "hit_chosen"):
            assert np.array_equal(g[k], o[k]), (k, np.nonzero(g[k] != o[k])[0][:5])
        pend, ost = s.get_instances(pending=True), orc.get_state()
        for k in ("b", "qr", "q", "S"):
            assert np.array_equal(pend[k], ost[k]), k
    return o


def _workload(I, R, seed=11):
    return W.generate(0, seed=seed, num_instances=I, window_requests=R, num_sessions=max(4, R // 6), cap_blocks=2048,
                      b_hi=8, b_max=64)


@pytest.mark.parametrize("I", [1, 31, 32, 33, 511, 512, 513, 1023, 1024, 1025, 2048])
def test_instance_counts(P, I):
    wl = _workload(I, 80)
    _check(P, wl.model, wl.instances, wl.window)


@pytest.mark.parametrize("R", [1, 2, 7, 8, 9, 32, 33, 34, 65, 130])
def test_window_lengths(P, R):
    wl = _workload(12, R)
    _check(P, wl.model, wl.instances, wl.window)


def _prompts(nb_of, chains, I):
    """Window of one prompt per entry of nb_of (tokens; chains[k] its blocks' hashes), empty caches."""
    off = np.zeros(len(chains) + 1, np.uint64)
    off[1:] = np.cumsum([c.size for c in chains])
    R = len(chains)
    win = W.Window(chain_off=off, chain_hash=np.concatenate(chains).astype(np.uint64),
                   prompt_tokens=np.array(nb_of, np.uint32), ttft_target=np.full(R, 1e7, np.float32),
                   tpot_target=np.full(R, 1e4, np.float32), session=np.zeros(R, np.uint32), out_tokens=np.zeros(R, np.uint32))
    z = np.zeros(I, np.int64)
    ins = W.Instances(b=z.astype(np.int32), qr=z.astype(np.int32), q=z, S=z.copy(), M_KV=np.full(I, 10 ** 8, np.int64),
                      B_max=np.full(I, 10 ** 5, np.int32), cap_blocks=np.full(I, 4096, np.uint64),
                      chain_inst=np.zeros(0, np.uint32), chain_off=np.zeros(1, np.uint64),
                      chain_hash=np.zeros(0, np.uint64), chain_parent=np.zeros(0, np.uint64))
    return ins, win


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("shorts", [31, 32, 33, 45, 130])
def test_prompts_without_a_block_hide_no_inserts(P, shorts, mode):
    """A chain cached by the window's first request, prompts too short for a block on the same instance, then
    requests that share half of that chain, from further back than the common prefixes reach."""
    rng = np.random.default_rng(3)
    new = lambda n: rng.integers(2, 2 ** 63, n, dtype=np.int64).astype(np.uint64)
    base = new(10)
    chains = [base] + [new(0)] * shorts + [np.concatenate([base[:5], new(3)]), base, new(4)]
    ins, win = _prompts([160] + [8] * shorts + [128, 160, 64], chains, 1)
    o = _check(P, dict(W.MODEL_DEFAULT), ins, win, mode)
    assert o["hit_chosen"][shorts + 1:].tolist() == [5, 10, 0]


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("I,R,seed", [(3, 400, 1), (70, 900, 2)])
def test_windows_of_mixed_prompt_lengths(P, I, R, seed, mode):
    rng = np.random.default_rng(seed)
    trunk = [rng.integers(2, 2 ** 63, 300, dtype=np.int64).astype(np.uint64) for _ in range(8)]
    lens, chains = [], []
    for _ in range(R):
        if rng.random() < 0.4:
            n, c = 0, np.zeros(0, np.uint64)
        else:
            t, cut = trunk[int(rng.integers(8))], int(rng.integers(1, 300))
            c = t[:cut]
            if rng.random() < 0.5:
                c = np.concatenate([c, rng.integers(2, 2 ** 63, int(rng.integers(1, 20)), dtype=np.int64).astype(np.uint64)])
            n = c.size
        chains.append(c)
        lens.append(16 * n + int(rng.integers(0, 16)))
    ins, win = _prompts(lens, chains, I)
    _check(P, dict(W.MODEL_DEFAULT), ins, win, mode)


@pytest.mark.parametrize("selector", range(6))
def test_equal_keys_go_to_the_lowest_instance(P, selector):
    # every instance in the same state and with the same cache: all keys of a row are equal at first
    wl = _workload(520, 60)
    ins = wl.instances
    for a in (ins.b, ins.qr, ins.q, ins.S):
        a[:] = a[0]
    ins.chain_inst, ins.chain_off = np.zeros(0, np.uint32), np.zeros(1, np.uint64)
    ins.chain_hash, ins.chain_parent = np.zeros(0, np.uint64), np.zeros(0, np.uint64)
    o = _check(P, dict(wl.model, selector=selector), ins, wl.window)
    assert o["assign"][0] == 0


@pytest.mark.parametrize("shift", ["kv_room", "tokens", "queue"])
def test_sums_beyond_32_bits(P, shift):
    # KV capacities, held tokens or queued tokens from which a 32-bit sum could overflow in the window
    wl = _workload(70, 90)
    ins = wl.instances
    ins.M_KV[:] = 1 << 45 if shift != "queue" else ins.M_KV
    if shift == "tokens":
        ins.S[::3] += (1 << 30) - 5000
        ins.S[1::3] += 1 << 40
    if shift == "queue":
        ins.q[::2] += (1 << 30) - 9000
        ins.q[5::7] += 1 << 35
    for sel in (0, 5):
        _check(P, dict(wl.model, selector=sel), ins, wl.window)


@pytest.mark.parametrize("M", [2 ** 30, 2 ** 31 - 1, 2 ** 31 + 5, 2 ** 45, 2 ** 50 - 1])
@pytest.mark.parametrize("below", [-16, -1, 0, 1, 400, 10 ** 6])
def test_kv_room_beyond_32_bits(P, M, below):
    """The window's tokens bound what an instance can gain, so rooms beyond 32 bits alone need no 64-bit sums;
    held and queued tokens a few tokens on either side of where the sums would leave 2^30."""
    wl = _workload(5, 60, seed=14)
    ins = wl.instances
    tokens = 16 * (int(wl.window.chain_off[-1]) + wl.window.R)
    ins.M_KV[:] = M
    ins.S[:4] = 2 ** 30 - tokens - below
    ins.q[2:] = 2 ** 30 - tokens - below
    ins.b[:], ins.qr[:] = 1, 0
    wl.window.tpot_target[:] = 1e9  # every request is admitted somewhere
    wl.window.ttft_target[:] = 1e9
    _check(P, dict(wl.model, eta=1e6), ins, wl.window)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("ablation", ["F", "C", "CT"])
@pytest.mark.parametrize("sel", range(6))
def test_pairs_that_a_rank_does_not_tell_apart(P, sel, ablation, mode):
    """A rank holds part of a key: here many pairs are equal in that part (hits and queues around the 8191 it
    stops at, few values of b, b and h of 0 under the D-C-Q fallback, negative headrooms where everything is
    admitted), so the rest of the key or the tie word decides."""
    from oracle import ABLATIONS
    rng = np.random.default_rng(sel)
    I, R = 120, 40
    trunk = rng.integers(2, 2 ** 63, 8300, dtype=np.int64).astype(np.uint64)
    ins, win = _prompts([16 * 8300 + 3] * R, [trunk] * R, I)
    ins.M_KV[:] = 2 ** 29
    ins.cap_blocks[:] = 8400
    ins.b[:] = rng.choice([0, 7], I)
    ins.qr[:] = rng.choice([0, 3, 8190, 8191, 8192, 9000, 131000], I)
    ins.B_max[:] = ins.b + ins.qr + 1  # each takes one request: every decision is the next in order
    n = rng.choice([0, 1, 8189, 8190, 8191, 8192, 8250], I)
    ins.chain_inst = np.arange(I, dtype=np.uint32)
    ins.chain_off = np.concatenate([[0], np.cumsum(n)]).astype(np.uint64)
    ins.chain_hash = np.concatenate([trunk[:k] for k in n])
    ins.chain_parent = np.zeros(I, np.uint64)
    win.tpot_target[::2] = 5.0  # missed: the fallback (or, with everything admitted, a negative headroom)
    model = dict(W.MODEL_DEFAULT, eta=1e6, b1=0.0)
    orc = Oracle(I, dict(model, selector=sel, **ABLATIONS[ablation])).load(ins)
    with P.Scheduler(I, ins.cap_blocks, R, int(win.chain_off[-1]), dict(model, selector=sel, **P.ABLATIONS[ablation]),
                     probe_mode=mode) as s:
        s.load_workload_instances(ins)
        g, o = s.schedule_window(win), orc.schedule(win)
        for k in ("assign", "path", "hit_chosen"):
            assert np.array_equal(g[k], o[k]), (k, np.nonzero(g[k] != o[k])[0][:5])
    assert set(o["path"].tolist()) == ({0} if ablation == "C" else {0, 1})


@pytest.mark.parametrize("I", [1, 33, 512, 513, 1024, 1025, 2048])
@pytest.mark.parametrize("sel", [0, 5])
def test_instance_counts_in_linear_mode(P, I, sel):
    """The linear kernels have an instance of their own per instances a thread (1, 2, 4); every cache here has
    holes, and hits that rise in the window end at one or go on past it."""
    wl = _workload(I, 80, seed=13)
    ins = wl.instances
    keep = np.random.default_rng(4).random(ins.chain_hash.size) > 0.03
    n = np.concatenate([[0], np.cumsum(keep)])[ins.chain_off.astype(np.int64)]
    ins.chain_hash, ins.chain_off = ins.chain_hash[keep], n.astype(np.uint64)
    _check(P, dict(wl.model, selector=sel), ins, wl.window, mode=0)


@pytest.mark.parametrize("sel,kv", [(0, 0), (5, 0), (0, 1 << 45)])
def test_caches_with_holes(P, sel, kv):
    """Caches that are not prefix-closed: hits that rise in the window go on through blocks the committed
    table holds past a hole, and end at a reserved hash."""
    wl = _workload(24, 150, seed=12)
    ins, win = wl.instances, wl.window
    rng = np.random.default_rng(2)
    off = [0]
    keep = rng.random(ins.chain_hash.size) > 0.02
    for c in range(ins.chain_inst.size):
        off.append(off[-1] + int(keep[int(ins.chain_off[c]):int(ins.chain_off[c + 1])].sum()))
    ins.chain_hash, ins.chain_off = ins.chain_hash[keep], np.array(off, np.uint64)
    # some blocks' hashes are the reserved 0, in every chain that holds them; the oracle, which reserves
    # no value, sees a hash of its own in each of those places
    zero = np.isin(win.chain_hash, rng.choice(win.chain_hash, 40))
    own = dict(vars(win), chain_hash=win.chain_hash.copy())
    own["chain_hash"][zero] = rng.integers(2, 2 ** 63, int(zero.sum()), dtype=np.int64).astype(np.uint64)
    win.chain_hash[zero] = 0
    owin = W.Window(**own)
    if kv:
        ins.M_KV[:] = kv
    model = dict(wl.model, selector=sel)
    orc = Oracle(ins.I, model).load(ins)
    with P.Scheduler(ins.I, ins.cap_blocks, win.R, int(win.chain_off[-1]), model, table_load_factor=0.5,
                     probe_mode=P.PS_PROBE_LINEAR) as s:
        s.load_workload_instances(ins)
        assert np.array_equal(s.score_window(win, want=("hits",))["hits"], orc.score_rows(owin)["hits"])
        g, o = s.schedule_window(win), orc.schedule(owin)
        for k in ("assign", "path", "hit_chosen"):
            assert np.array_equal(g[k], o[k]), (k, np.nonzero(g[k] != o[k])[0][:5])
