"""Cases of the scheduler's performance measurements: what a program that uses this library has it do.

A gateway keeps one scheduler context per instance pool.  It hands over windows of requests (one request
at a time when traffic is low, thousands when it is not), reads the decisions, commits them and lets the
engines' progress and the eviction run between windows; diagnostics ask for every pair's score; a pool
that spans several contexts is scored in column blocks; a restarted scheduler loads its caches first.

Inputs are drawn on the GPU from a seed: sessions resend their history with every step (a request's chain
extends the session's previous one), all share a system prompt, each session's history is cached on its
home instance and a part of it on another, and every cache is filled up with other chains.

Results are exact: hits, classes, picks and states are whole numbers, and the predicted latencies are
IEEE single precision in the operation order that include/packserve.h lays down, so another correct
implementation gives the same bits.
"""
import math

import numpy as np
import torch

import paper_2609_33224_gb300 as P

MODEL = dict(a0=5.0, a1=0.02, a2=1e-6, a3=1e-6, a4=0.0, a5=0.0, b0=8.0, b1=0.15, b2=2e-5, g_q=0.004, eta=0.5,
             lout_median=556.0, interference_mode=0, ttft_filter=1, seg_lo=[0], ema_factor=[1.0])
MODELS = {
    "default": MODEL,
    # Eq. 9 of the paper with factors that online calibration has learned per decode-batch segment
    "eq9": dict(MODEL, interference_mode=1, seg_lo=[0, 17, 65], ema_factor=[1.0, 1.0625, 1.125]),
    # smallest predicted headroom first (Table 4's H-C-Q order)
    "hcq": dict(MODEL, selector=5),
    # Algorithm 1 without the optional TTFT test
    "algorithm1": dict(MODEL, ttft_filter=0),
}
STREAM_WINDOWS = 512  # windows of new requests a streaming state holds
ALL = ("hits", "tpot", "ttft", "cls", "best", "path")

_BASE = dict(kind="schedule", instances=64, requests=64, sessions=64, zipf=0.0, ctx_lo=4096, ctx_hi=131072, sys=4096,
             cache=8192, fill=1.0, load_factor=0.5, probe="search", inputs="device", spare=1, b_hi=64, q_hi=8192,
             tpot=50.0, ttft=2000.0, model="default")


def _case(**kw):
    return dict(_BASE, **kw)


def listed():
    return [
        # the smallest diagnostic call: every pair's score of a tiny window
        _case(name="score_8x64", kind="score", instances=8, requests=64, sessions=4, ctx_lo=1024, ctx_hi=8192, sys=0,
              cache=4096, fill=0.75, b_hi=32),
        # a gateway at low traffic: one request arrives, on a context that can also take bursts of 64
        _case(name="route_1_request", instances=64, requests=1, sessions=512, ctx_lo=8192, inputs="host", spare=64,
              cache=65536),
        # arrivals of some 20 ms, pool size and window not round, shared-prefix form from pinned memory
        _case(name="schedule_201x117_tree", instances=201, requests=117, sessions=96, inputs="tree", spare=4, cache=30001,
              b_hi=128, tpot=80.0, model="algorithm1"),
        # evaluation scale, resident inputs: packing and fallback both occur
        _case(name="schedule_64x4096", instances=64, requests=4096, sessions=512, ctx_lo=8192, cache=200000, b_hi=128),
        # production scale, resident inputs: long queues, most decisions by the cache-aware fallback
        _case(name="schedule_1024x16384", instances=1024, requests=16384, sessions=8192, zipf=1.1, cache=200000,
              load_factor=0.9, b_hi=128, q_hi=32768, ttft=3000.0),
        # production scale, short queues and a loose target (most decisions packed), shared-prefix windows
        _case(name="schedule_999x3001_tree", instances=999, requests=3001, sessions=2048, zipf=1.1, inputs="tree",
              cache=40000, load_factor=0.9, b_hi=128, q_hi=4096, tpot=200.0, ttft=3000.0),
        # long contexts: 128K to 1M tokens a prompt, 32K of them shared
        _case(name="schedule_256x512_long", instances=256, requests=512, sessions=384, ctx_lo=131072, ctx_hi=1048576,
              sys=32768, cache=262144, b_hi=128, q_hi=16384, tpot=80.0, ttft=3000.0),
        # production scale, every pair's score kept on the device
        _case(name="score_1024x16384", kind="score", instances=1024, requests=16384, sessions=8192, zipf=1.1,
              cache=200000, load_factor=0.9, b_hi=128, q_hi=32768, ttft=3000.0),
        # caches that are not closed under prefixes (blocks dropped one by one): the linear probe, decisions and scores
        _case(name="linear_100x300", kind="linear", instances=100, requests=300, sessions=64, ctx_lo=2048, ctx_hi=32768,
              probe="linear", cache=16384, b_hi=64, tpot=80.0, model="eq9"),
        # one column block of a pool that spans several contexts
        _case(name="shard_512x4096", kind="shard", instances=512, requests=4096, sessions=2048, zipf=1.1, cache=32768,
              b_hi=128, q_hi=4096, tpot=200.0, model="hcq"),
        # a streaming gateway's window: decisions, commit, engine progress, eviction
        _case(name="stream_1024x500", kind="stream", instances=1024, requests=500, sessions=8192, zipf=1.1, cache=200000,
              b_hi=32, q_hi=8192, tpot=100.0, ttft=3000.0),
        # a scheduler starts: a new context loads every instance's cache
        _case(name="load_96x20000", kind="load", instances=96, requests=32, sessions=256, cache=20000, b_hi=64),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["score", "score", "schedule", "schedule", "schedule", "schedule", "linear", "shard", "stream",
                       "load"])
    I = log(8, 1500) if kind in ("score", "schedule", "shard") else log(16, 256)
    ctx_lo = rng.choice([1024, 4096, 8192, 32768])
    ctx_hi = ctx_lo * rng.choice([4, 8, 16, 32])
    mean_blocks = (ctx_lo + 0.4 * (ctx_hi - ctx_lo)) / 16
    R = log(1, 8192) if kind in ("score", "schedule", "shard") else log(16, 400)
    R = max(1, min(R, int(6e6 / I), int(2e7 / mean_blocks)))
    if kind == "stream":
        R = max(8, min(R, int(3e5 / mean_blocks)))
    cache = min(log(2000, 200000), int(2e7 / I))
    if kind == "load":
        cache = min(cache, 40000)
    sys = rng.choice([0, 1024, 4096])
    cache = max(cache, 2 * sys // 16 + 64)
    q_hi = rng.choice([1024, 4096, 8192, 32768])
    return _case(kind=kind, instances=I, requests=R, sessions=max(2, log(max(2, R / 8), 4 * R + 8)), zipf=rng.choice([0.0, 1.1]),
                 ctx_lo=ctx_lo, ctx_hi=ctx_hi, sys=sys, cache=cache, fill=1.0 if kind == "stream" else rng.choice([0.6, 0.9, 1.0]),
                 load_factor=0.5 if kind == "stream" else rng.choice([0.5, 0.75, 0.9]),
                 probe="linear" if kind == "linear" else "search",
                 inputs=rng.choice(["device", "host", "tree"]) if kind in ("score", "schedule") else "device",
                 spare=rng.choice([1, 1, 3]), b_hi=rng.choice([32, 64, 128]), q_hi=q_hi,
                 tpot=rng.choice([50.0, 80.0, 200.0]), ttft=rng.choice([2000.0, 3000.0]),
                 model=rng.choice(["default", "default", "eq9", "hcq", "algorithm1"]))


# ---- inputs ---------------------------------------------------------------------------------------------

def _s64(x):
    x &= (1 << 64) - 1
    return x - (1 << 64) if x >= 1 << 63 else x


def _lsr(x, k):
    return (x >> k) & ((1 << (64 - k)) - 1)


def _hash(branch, pos, seed):
    """64-bit block hash of position pos of a token branch (never 0 or all ones)."""
    x = branch * _s64(0xD6E8FEB86659FD93) + pos * _s64(0xA0761D6478BD642F) + _s64(seed * 0xE7037ED1A0B428DB + 1)
    x = (x ^ _lsr(x, 30)) * _s64(0xBF58476D1CE4E5B9)
    x = (x ^ _lsr(x, 27)) * _s64(0x94D049BB133111EB)
    x = x ^ _lsr(x, 31)
    return torch.where((x == 0) | (x == -1), torch.full_like(x, 7), x)


_FILL = 1 << 40  # branch ids of the chains that fill the caches up


def _csr(lens):
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device=lens.device)
    torch.cumsum(lens, 0, out=off[1:])
    return off


def _flat(branch, first, lens, sysb, seed):
    """Chains laid end to end: chain c covers positions first[c] .. first[c] + lens[c] of its branch; positions
    below sysb belong to the shared system prompt (branch 0)."""
    off = _csr(lens)
    out = torch.empty(int(off[-1]), dtype=torch.int64, device=lens.device)
    n, lo = lens.numel(), 0
    while lo < n:  # in pieces, so that the index arrays stay small
        hi = int(torch.searchsorted(off, off[lo] + (1 << 25), right=True)) - 1
        hi = min(n, max(hi, lo + 1))
        a, b = int(off[lo]), int(off[hi])
        c = torch.repeat_interleave(torch.arange(lo, hi, device=lens.device), lens[lo:hi], output_size=b - a)
        pos = torch.arange(a, b, device=lens.device) - (off[c] - first[c])
        out[a:b] = _hash(torch.where(pos < sysb, 0, branch[c]), pos, seed)
        lo = hi
    return off, out


def _requests(c, n, g, dev):
    """n requests in arrival order: session, epoch (token branch within the session), prompt tokens, and the
    latest earlier request whose prompt it extends (-1: none); and every session's prompt length before them."""
    S = c["sessions"]
    lo = max(c["ctx_lo"], c["sys"] + 64)  # every prompt goes on after the system prompt
    span = c["ctx_hi"] - lo
    if c["zipf"]:
        ses = torch.multinomial((torch.arange(S, device=dev) + 1.0).pow(-c["zipf"]), n, replacement=True, generator=g)
    else:
        ses = torch.randint(S, (n,), device=dev, generator=g)
    start = torch.randint(span // 2, (S,), device=dev, generator=g)
    inc = torch.exp(torch.randn(n, device=dev, generator=g) * 0.8 + 7.5).clamp_(16, max(32, span // 4)).to(torch.int64)
    order = torch.argsort(ses, stable=True)
    so, grown = ses[order], torch.cumsum(inc[order], 0)
    head = torch.searchsorted(so, so)  # first place of each session's run
    x = torch.empty_like(inc)
    x[order] = start[so] + grown - (grown[head] - inc[order][head])
    epoch = torch.div(x, span, rounding_mode="floor")
    L = lo + x - epoch * span
    prev = torch.full_like(ses, -1)
    same = (so[1:] == so[:-1]) & (epoch[order][1:] == epoch[order][:-1])
    prev[order[1:]] = torch.where(same, order[:-1], -1)
    return ses, epoch, L, prev, lo + start


def _branch(ses, epoch):
    return 1 + ses * 4096 + torch.clamp(epoch, max=4095)


def _caches(c, start, g, dev):
    """Which part of which session every instance caches: (session, instance, blocks, hole) with the blocks
    counted from the chain's start and hole the block that is missing (linear mode; -1: none)."""
    I, S, sysb = c["instances"], c["sessions"], c["sys"] // 16
    home = torch.randint(I, (S,), device=dev, generator=g)
    other = (home + 1 + torch.randint(max(1, I - 1), (S,), device=dev, generator=g)) % I
    part = (start // 16).float() * (0.2 + 0.8 * torch.rand(S, device=dev, generator=g))
    ses = torch.arange(S, device=dev)
    ses, inst = torch.cat([ses, ses]), torch.cat([home, other])
    blk = torch.cat([start // 16, part.to(torch.int64)])
    keep = (blk > sysb + 1) & (torch.cat([torch.ones(S, device=dev), torch.rand(S, device=dev, generator=g)]) > 0.4)
    if I == 1:
        keep[S:] = False
    ses, inst, blk = ses[keep], inst[keep], blk[keep]
    # what fits: 90% of an instance's blocks at most
    order = torch.argsort(inst, stable=True)
    ses, inst, blk = ses[order], inst[order], blk[order]
    own = blk - sysb
    run = torch.cumsum(own, 0)
    head = torch.searchsorted(inst, inst)
    fits = run - (run[head] - own[head]) <= int(0.9 * c["fill"] * c["cache"]) - sysb
    ses, inst, blk = ses[fits], inst[fits], blk[fits]
    hole = torch.full_like(blk, -1)
    if c["probe"] == "linear":
        at = sysb + (torch.rand(blk.numel(), device=dev, generator=g) * (blk - sysb - 1)).to(torch.int64)
        hole = torch.where(torch.rand(blk.numel(), device=dev, generator=g) < 0.5, at, hole)
    return ses, inst, blk, hole


def _chains(c, placed, seed, dev):
    """The caches as chains: (instance, offsets, hashes, parent hash, age group); parents come first."""
    I, sysb = c["instances"], c["sys"] // 16
    ses, inst, blk, hole = placed
    zero = torch.zeros_like
    ids = torch.arange(I, device=dev)
    br, sysv = _branch(ses, zero(ses)), torch.full_like(ses, sysb)
    cut = torch.where(hole >= 0, hole, blk)
    used = sysb + torch.zeros(I, dtype=torch.int64, device=dev).index_add_(0, inst, blk - sysb - (hole >= 0).to(torch.int64))
    need = torch.clamp(int(c["fill"] * c["cache"]) - used, min=0)
    flen = 512 if c["cache"] > 16384 else 96
    nf = (need + flen - 1) // flen
    finst = torch.repeat_interleave(ids, nf)
    fk = torch.arange(finst.numel(), device=dev) - _csr(nf)[finst]
    flens = torch.clamp(need[finst] - fk * flen, max=flen)
    tail = hole >= 0
    who = torch.cat([ids, inst, inst[tail], finst])
    branch = torch.cat([zero(ids), br, br[tail], _FILL + torch.arange(finst.numel(), device=dev)])
    first = torch.cat([zero(ids), sysv, hole[tail] + 1, torch.full_like(finst, sysb)])  # not the system prompt's blocks
    lens = torch.cat([torch.full_like(ids, sysb), cut - sysb, (blk - hole - 1)[tail], flens])
    at = first - 1
    parent = torch.where((at >= 0) & (branch < _FILL), _hash(torch.where(at < sysb, 0, branch), at, seed), 0)
    # age: the filling chains spread over all ages, oldest first; sessions and the system prompt are recent
    age = torch.cat([torch.full_like(ids, 31), 24 + ses % 7, 24 + ses[tail] % 7, _lsr(_hash(branch[-finst.numel():], 0, seed), 8) % 28
                     if finst.numel() else finst])
    keep = lens > 0
    who, branch, first, lens, parent, age = (t[keep] for t in (who, branch, first, lens, parent, age))
    return who, branch, first, lens, parent, age


class _Window:
    pass


def _window(c, ses, epoch, L, prev, seed, dev, inputs, out=None):
    """The window in the form the case asks for: resident, or host arrays whole or with parent links."""
    n, sysb = L.numel(), c["sys"] // 16
    nb, br = L // 16, _branch(ses, epoch)
    w = _Window()
    first = torch.where(prev >= 0, nb[prev.clamp(min=0)], 0) if inputs == "tree" else torch.zeros_like(nb)
    off, hashes = _flat(br, first, nb - first, sysb, seed)
    arrays = dict(chain_off=off, chain_hash=hashes, prompt_tokens=L.to(torch.int32),
                  ttft_target=torch.full((n,), c["ttft"], device=dev), tpot_target=torch.full((n,), c["tpot"], device=dev))
    if inputs == "tree":
        arrays["parent"] = prev.to(torch.int32)
    if out is not None:
        arrays["out_tokens"] = out.to(torch.int32)
    for k, v in arrays.items():
        if inputs == "host":  # an ordinary program's numpy arrays
            v = v.cpu().numpy()
            v = v.view({"int64": np.uint64, "int32": np.uint32}.get(v.dtype.name, v.dtype))
        elif inputs == "tree":
            v = v.cpu().pin_memory()
        setattr(w, k, v)
    w.blocks = int(nb.sum())
    return w


def _draw_inputs(case, seed):
    c = dict(_BASE, **case)
    dev = torch.device("cuda", 0)
    g = torch.Generator(device=dev)
    g.manual_seed(seed * 1000003 + 17)
    n = c["requests"] * (STREAM_WINDOWS if c["kind"] == "stream" else 1)
    ses, epoch, L, prev, start = _requests(c, n, g, dev)
    placed = _caches(c, start, g, dev)
    r = np.random.RandomState(seed % (1 << 32))
    I = c["instances"]
    M = 16 * c["cache"]
    st = dict(b=r.randint(0, c["b_hi"] + 1, I).astype(np.int32), q=r.randint(0, c["q_hi"] + 1, I).astype(np.int64))
    st["qr"] = ((st["q"] + 4095) // 4096).astype(np.int32)
    st["B_max"] = np.full(I, 2 * c["b_hi"], np.int32)
    mean = c["ctx_lo"] + (c["ctx_hi"] - c["ctx_lo"]) // 4
    st["S"] = np.minimum(st["b"].astype(np.int64) * mean, M * st["b"].astype(np.int64) // (2 * c["b_hi"]))
    # room for the longest prompt also where the cache is small beside it
    st["M_KV"] = np.full(I, max(M, int(1.5 * c["ctx_hi"])), np.int64)
    return c, dev, g, (ses, epoch, L, prev), placed, st


def _make_scheduler(c, max_requests, max_blocks, **kw):
    return P.Scheduler(c["instances"], np.full(c["instances"], c["cache"], np.uint64), max_requests, max_blocks,
                       MODELS[c["model"]], table_load_factor=c["load_factor"],
                       probe_mode=P.PS_PROBE_LINEAR if c["probe"] == "linear" else P.PS_PROBE_SEARCH, **kw)


def _load_caches(c, s, placed, seed, dev, by_age=False):
    who, branch, first, lens, parent, age = _chains(c, placed, seed, dev)
    # parents first: with ages, the system prompt and the sessions' chains, then the rest from old to new
    groups = [age >= 31, (age >= 24) & (age < 31)] + [age == a for a in range(24)] if by_age else [torch.ones_like(age, dtype=torch.bool)]
    stamps = [31, 30] + list(range(24)) if by_age else [0]
    for sel, stamp in zip(groups, stamps):
        if not bool(sel.any()):
            continue
        off, hashes = _flat(branch[sel], first[sel], lens[sel], c["sys"] // 16, seed)
        who_s, parent_s = who[sel].to(torch.int32), parent[sel].contiguous()
        torch.cuda.synchronize()
        s.insert_chains(who_s, off, hashes, parent_s, last_use=stamp)


def prepare(case, seed):
    c, dev, g, (ses, epoch, L, prev), placed, st = _draw_inputs(case, seed)
    R, longest = c["requests"], c["ctx_hi"] // 16 + 1
    if c["kind"] == "load":
        who, branch, first, lens, parent, _ = _chains(c, placed, seed, dev)
        off, hashes = _flat(branch, first, lens, c["sys"] // 16, seed)
        host = [t.cpu().numpy() for t in (who.to(torch.int32), off, hashes, parent)]
        return dict(case=c, chains=[host[0].view(np.uint32)] + [h.view(np.uint64) for h in host[1:]], state=st)
    if c["kind"] == "stream":
        # decoding and queued requests that the engines hold when the stream is joined
        r = np.random.RandomState((seed + 1) % (1 << 32))
        nd, nq = st["b"], np.minimum(st["qr"], 3)
        inst = np.concatenate([np.repeat(np.arange(c["instances"]), nd), np.repeat(np.arange(c["instances"]), nq)])
        state = np.concatenate([np.ones(nd.sum(), np.uint32), np.zeros(nq.sum(), np.uint32)])
        out = np.clip(np.exp(r.normal(5.0, 0.6, inst.size)), 16, 4096).astype(np.uint32)
        room = np.maximum(1024, (st["M_KV"] // (2 * c["b_hi"]))[inst])
        Lr = np.minimum(r.randint(c["ctx_lo"], c["ctx_hi"], inst.size), room).astype(np.uint32)
        rem = np.where(state == 1, 1 + r.randint(0, 1 << 30, inst.size) % out, r.randint(256, 4096, inst.size)).astype(np.uint64)
        s = _make_scheduler(c, R, longest * R, track_lru=True, max_active_requests=4 * c["b_hi"] + 64)
        _load_caches(c, s, placed, seed, dev, by_age=True)
        s.load_instances(st["b"], st["qr"], st["q"], st["S"], st["M_KV"], st["B_max"])
        s.load_requests(dict(inst=inst, state=state, L=Lr, out=out, rem=rem))
        outs = torch.exp(torch.randn(L.numel(), device=dev, generator=g) * 0.6 + 5.0).clamp_(16, 4096)
        wins = [_window(c, ses[a:a + R], epoch[a:a + R], L[a:a + R], prev[a:a + R], seed, dev, "device", outs[a:a + R])
                for a in range(0, L.numel(), R)]
        return dict(case=c, s=s, windows=wins, step=0)
    w = _window(c, ses, epoch, L, prev, seed, dev, c["inputs"])
    s = _make_scheduler(c, R * c["spare"], w.blocks if c["spare"] == 1 else longest * R * c["spare"])
    _load_caches(c, s, placed, seed, dev)
    s.load_instances(st["b"], st["qr"], st["q"], st["S"], st["M_KV"], st["B_max"])
    return dict(case=c, s=s, window=w)


# ---- one pass -------------------------------------------------------------------------------------------

def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "schedule":
        d = state["s"].schedule_window(state["window"], device_outputs=c["inputs"] == "device")
        if c["requests"] > 1:  # the gateway's own records follow the window; a single request's it updates itself
            d["instances"] = state["s"].get_instances(pending=True)
        return d
    if kind == "score":
        return state["s"].score_window(state["window"], want=ALL, device_outputs=True)
    if kind == "linear":
        return state["s"].schedule_window(state["window"], scores=ALL, device_outputs=True)
    if kind == "shard":
        s, w = state["s"], state["window"]
        wmin = s.shard_wmin(w, device_outputs=True)
        # the pool's minimum over all blocks would come from an all-reduce here; this block stands alone
        return dict(s.shard_pick(wmin, 0, scores=ALL, device_outputs=True), wmin=wmin)
    if kind == "stream":
        s, k = state["s"], state["step"]
        state["step"] = k + 1
        d = s.schedule_window(state["windows"][k % STREAM_WINDOWS], device_outputs=True)
        s.commit_window(last_use=32 + k)
        s.advance_window(200.0, 16000, evict=True)
        return dict(d, cached=s.cached_blocks().astype(np.int64), instances=s.get_instances())
    # load: a scheduler starts and takes over the pool's caches and state
    st = state["state"]
    with _make_scheduler(c, c["requests"], c["requests"] * (c["ctx_hi"] // 16 + 1)) as s:
        s.insert_chains(*state["chains"])
        s.load_instances(st["b"], st["qr"], st["q"], st["S"], st["M_KV"], st["B_max"])
        return dict(cached=s.cached_blocks().astype(np.int64), instances=s.get_instances())


def work(case):
    c = dict(_BASE, **case)
    I, R = c["instances"], c["requests"]
    pairs, blocks = I * R, R * (c["ctx_lo"] + 0.3 * (c["ctx_hi"] - c["ctx_lo"])) / 16
    if c["kind"] == "load":  # every chain block read and its slot written
        return {"bytes": 16.0 * I * c["fill"] * c["cache"], "flops": 0.0}
    scores = {"score": 13, "linear": 13, "shard": 13}.get(c["kind"], 0)  # hit, TPOT, TTFT, class of a pair
    n = 8.0 * blocks + 21.0 * R + 72.0 * I + scores * pairs + 9.0 * R
    if c["kind"] == "stream":  # the admitted blocks' slots and metadata, written once and evicted once
        n += 2 * 24.0 * 0.3 * blocks
    return {"bytes": n, "flops": 24.0 * pairs}


def tolerance(case):
    # Two runs, two builds and the single-threaded restatement under oracle/ agree in every bit: the order of the
    # single-precision operations is part of the interface, everything else is whole numbers.
    return "exact"


def exact(case, seed):
    """Scores in 64 bits from the way the inputs were drawn: hits, TPOT and TTFT (Eq. 4 to 9)."""
    c, dev, g, (ses, epoch, L, prev), placed, st = _draw_inputs(case, seed)
    if c["kind"] not in ("score", "linear", "shard"):
        return None  # whole numbers only
    m, I, sysb = MODELS[c["model"]], c["instances"], c["sys"] // 16
    pses, pinst, blk, hole = placed
    depth = torch.full((c["sessions"], I), sysb, dtype=torch.int64, device=dev)
    depth[pses, pinst] = torch.where(hole >= 0, hole, blk)
    nb = (L // 16)[:, None]
    hits = torch.minimum(torch.where((epoch == 0)[:, None], depth[ses], sysb), nb)
    n, cached = (L[:, None] - 16 * hits).double(), (16 * hits).double()
    t = {k: torch.from_numpy(np.asarray(v)).to(dev)[None, :].double() for k, v in st.items()}
    f64 = {k: float(np.float32(m[k])) for k in ("a0", "a1", "a2", "a3", "a4", "a5", "b0", "b1", "b2", "g_q", "lout_median")}
    tpf = f64["a0"] + f64["a1"] * n + f64["a2"] * n * cached + f64["a3"] * n * n + f64["a4"] * cached + f64["a5"] * cached * cached
    B, S = t["b"] + t["qr"] + 1, t["S"] + L[:, None].double()
    seg = torch.bucketize(B, torch.tensor(m["seg_lo"], dtype=torch.float64, device=dev), right=True) - 1
    dec = (f64["b0"] + f64["b1"] * B + f64["b2"] * S) * torch.tensor(m["ema_factor"], dtype=torch.float64, device=dev)[seg]
    if m["interference_mode"] == 0:
        tpot = dec + f64["g_q"] * (t["q"] + n)
    else:
        tpot = dec + torch.where(B > 1, tpf / max(1.0, f64["lout_median"]), torch.zeros_like(tpf))
    ttft = tpf + f64["a0"] * t["qr"] + f64["a1"] * t["q"]
    # classes and picks follow from comparisons of the rounded latencies: no 64-bit value stands for them
    scores = dict(hits=hits.to(torch.int32), tpot=tpot, ttft=ttft, cls=None, best=None, path=None)
    if c["kind"] == "score":
        return scores
    if c["kind"] == "shard":
        return dict(key=None, tie=None, scores=scores, wmin=None)
    return dict(assign=None, path=None, hit_chosen=None, scores=scores)
