"""What a pending window keeps until it is committed: its own chains, offsets, lengths and output
lengths, whatever is scored in between and whatever memory either window is in.

After each commit the state, the cache sizes, the cache contents (hit lengths) and the engines' next
step must equal those of an oracle that scheduled the same window with nothing in between."""
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


class _Device:
    """A window's arrays as CUDA tensors."""

    def __init__(self, win):
        import torch
        signed = {"uint64": np.int64, "uint32": np.int32}
        for k in ("chain_off", "chain_hash", "prompt_tokens", "ttft_target", "tpot_target", "out_tokens"):
            a = np.ascontiguousarray(getattr(win, k))
            setattr(self, k, torch.from_numpy(a.view(signed.get(a.dtype.name, a.dtype)).copy()).cuda())


FORMS = {"host": lambda w: w, "tree": W.tree_window, "device": _Device}
LARGE, SMALL = 1500, 40  # requests: more and less than the small-window staging block holds, in both host forms


@pytest.mark.parametrize("call", ["score_window", "shard_wmin"])
@pytest.mark.parametrize("form_b,R_b", [("host", 7), ("host", SMALL + 9), ("host", LARGE), ("host", 0), ("tree", 7),
                                        ("tree", LARGE), ("device", SMALL)])
@pytest.mark.parametrize("form_a,R_a", [("host", SMALL), ("host", LARGE), ("tree", LARGE), ("device", SMALL)])
def test_scoring_leaves_the_pending_window_alone(P, form_a, R_a, form_b, R_b, call):
    wl = W.generate(0, seed=21, num_instances=9, window_requests=R_a, num_sessions=30, cap_blocks=6000, b_max=2000)
    ins, A = wl.instances, wl.window
    ins.M_KV[:] = 10 ** 8
    B = wl.next_window(R_b) if R_b else W.Window(
        **{k: (v[:1] if k == "chain_off" else v[:0]) for k, v in vars(A).items()})
    if R_a == LARGE:
        assert W.tree_window(A).chain_hash.nbytes > 1 << 20
    orc = Oracle(ins.I, wl.model, track_lru=True).load(ins)
    req = wl.initial_requests()
    orc.load_requests(req)
    want_b = orc.score_rows(B)
    o = orc.schedule(A, window_id=1, streaming=True)
    blocks = max(int(A.chain_off[-1]), int(B.chain_off[-1]))
    with P.Scheduler(ins.I, ins.cap_blocks, LARGE + 9, blocks, wl.model, table_load_factor=0.02, track_lru=True,
                     max_active_requests=2048) as s:
        s.load_workload_instances(ins)
        s.load_requests(req)
        win_a, win_b = FORMS[form_a](A), FORMS[form_b](B)
        g = s.schedule_window(win_a)
        for k in ("assign", "path", "hit_chosen"):
            assert np.array_equal(g[k], o[k]), k
        pend = s.get_instances(pending=True)
        if call == "score_window":
            got_b = s.score_window(win_b)
            for k in ("hits", "cls", "best", "path"):
                assert np.array_equal(got_b[k], want_b[k]), k
        else:
            s.shard_wmin(win_b)
        for k, v in s.get_instances(pending=True).items():
            assert np.array_equal(v, pend[k]), k
        s.commit_window(last_use=1)
        assert [int(x) for x in s.cached_blocks()] == [orc.cached_blocks(i) for i in range(ins.I)]
        assert np.array_equal(s.score_window(A, want=("hits",))["hits"], orc.score_rows(A)["hits"])
        s.advance_window(40.0, 20000, evict=False)
        orc.advance(40.0, 20000, evict=False)
        st, ost = s.get_instances(), orc.get_state()
        for k in ("b", "qr", "q", "S"):
            assert np.array_equal(st[k], ost[k]), k
        # the next window finds the delta table empty
        g, o = s.schedule_window(win_b), orc.schedule(B, window_id=2, streaming=True)
        for k in ("assign", "path", "hit_chosen"):
            assert np.array_equal(g[k], o[k]), k


@pytest.mark.parametrize("mode", [0, 1])
def test_empty_windows_leave_the_state_as_it_is(P, mode):
    """A gateway whose interval holds no arrival: the pending state of an empty window is the committed one, on
    a new context, after other windows and after the engines' progress."""
    wl = W.generate(0, seed=22, num_instances=5, window_requests=40, num_sessions=12, cap_blocks=9000)
    ins, A = wl.instances, wl.window
    ins.M_KV[:] = 10 ** 8  # requests are admitted
    empty = W.Window(**{k: (v[:1] if k == "chain_off" else v[:0]) for k, v in vars(A).items()})
    orc = Oracle(ins.I, wl.model, track_lru=True).load(ins)
    with P.Scheduler(ins.I, ins.cap_blocks, 64, int(A.chain_off[-1]) * 2, wl.model, probe_mode=mode, track_lru=True,
                     max_active_requests=512) as s:
        s.load_workload_instances(ins)

        def nothing_arrives(win):
            before = s.get_instances()
            assert s.schedule_window(win)["assign"].size == 0
            for state in (s.get_instances(pending=True), s.commit_window() or s.get_instances()):
                for k, v in before.items():
                    assert np.array_equal(state[k], v), k

        nothing_arrives(empty)
        assert s.probe_stats()["greedy_fast"] == 0
        orc.load_requests(wl.initial_requests())
        s.load_requests(wl.initial_requests())
        nothing_arrives(_Device(empty))
        for w, win in enumerate((A, wl.next_window(40))):
            g, o = s.schedule_window(win), orc.schedule(win, window_id=w + 1, streaming=True)
            for k in ("assign", "path", "hit_chosen"):
                assert np.array_equal(g[k], o[k]), k
            assert (g["assign"] >= 0).any()
            assert s.probe_stats()["greedy_fast"] == (40 if mode else 0)
            s.commit_window(last_use=w + 1)
            nothing_arrives(empty)
            assert s.probe_stats()["greedy_fast"] == 0  # decisions of the last call: none
            s.advance_window(40.0, 20000, evict=False)
            orc.advance(40.0, 20000, evict=False)
            nothing_arrives(empty)
            st, ost = s.get_instances(), orc.get_state()
            for k in ("b", "qr", "q", "S"):
                assert np.array_equal(st[k], ost[k]), k


@pytest.mark.parametrize("form_a", ["host", "device"])
@pytest.mark.parametrize("blocks", [3, 200000])  # a small call goes through the staging block
def test_inserting_leaves_the_pending_window_alone(P, form_a, blocks):
    wl = W.generate(0, seed=23, num_instances=6, window_requests=SMALL, num_sessions=10, cap_blocks=6000)
    ins, A = wl.instances, wl.window
    ins.M_KV[:] = 10 ** 8
    ins.cap_blocks[:] = 300000
    chain = np.random.default_rng(6).integers(2, 2 ** 63, blocks, dtype=np.int64).astype(np.uint64)
    orc = Oracle(ins.I, wl.model, track_lru=True).load(ins)
    o = orc.schedule(A, window_id=1)
    orc.insert_chain(2, chain, last_use=1)
    with P.Scheduler(ins.I, ins.cap_blocks, SMALL, int(A.chain_off[-1]), wl.model, track_lru=True) as s:
        s.load_workload_instances(ins)
        win = FORMS[form_a](A)
        g = s.schedule_window(win)
        s.insert_blocks(2, chain, last_use=1)
        s.commit_window(last_use=1)
        for k in ("assign", "path", "hit_chosen"):
            assert np.array_equal(g[k], o[k]), k
        assert [int(x) for x in s.cached_blocks()] == [orc.cached_blocks(i) for i in range(ins.I)]
        assert np.array_equal(s.score_window(A, want=("hits",))["hits"], orc.score_rows(A)["hits"])
        st, ost = s.get_instances(), orc.get_state()
        for k in ("b", "qr", "q", "S"):
            assert np.array_equal(st[k], ost[k]), k
