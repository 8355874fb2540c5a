// Greedy in-window assignment (Algorithm 1 applied to the window's requests in arrival order).
//
// The paper's gateway decides each request online and updates the instance records along the
// request path before the next decision (Section 4, Metadata service; Section 7).  greedy_pipe_kernel
// replays that sequence for a whole window on the GPU: a pipelined cooperative launch of one deciding
// block, insert blocks and probe blocks.  Committed tables are never written here; the decisions and
// the updated state are a pending window that ps_commit_window applies.
#include "greedy_grid.h"
#include "ps_internal.cuh"

namespace {

// ----------------------------------------------------------------------------------------------
// The hit of a request is the first chain position not cached.  Chained block hashes make "block k
// equal" stand for "blocks 0..k equal", and an earlier request of the window has its whole chain cached
// on its instance, so with
//     M(s, i) = max lcp(s, t) over the earlier requests t of the window that went to i
// every position below M is cached on i while request s is decided, and from M on only the committed
// table counts:
//     hit(s, i) = hit0(s, i) if M <= hit0, else the first miss of main_i at or after M,
// which on a prefix-closed cache (the probe's search mode) is M itself.  Requests up to s - kLag count
// through the window's delta table, the later ones through their common prefixes with s (from the
// relations pass).
//
//   Deciding block (block 0).  Decides the requests in arrival order and publishes each decision as a
//   job (described at its section below).  No table access is on its per-request path, except where a
//   cache is not prefix-closed (LIN) and a hit rises past hit0.
//   Insert blocks.  Groups of kInsertGroup blocks take the jobs round-robin; a group's members split
//   each job's chain blocks between them, insert them into the delta table for the job's instance and
//   count the job done.  On prefix-closed caches the blocks chain[h, nb) do; else the whole chain goes
//   in, so that "block k of s is in the table for i" is exactly k < M and can be searched.
//   Probe blocks.  Take the rows round-robin.  For row s they wait until the jobs <= s - kLag are
//   done, replay those jobs (which instances have window inserts, where their last chain ended,
//   which instances took s's ancestors), then per instance start from hit0, raise the position to
//   the end of an ancestor's chain on the instance that took it (its chain is a prefix of s's, and
//   its inserts are in), probe the delta table there when the instance has window inserts, hand the
//   instances whose block is present to a warp search over the delta (LIN: then a walk of the main
//   table), and release the row's ready flag.  On prefix-closed caches the main table is never probed
//   here: positions past hit0 are absent from it.  Inserts of requests s - kLag + 1 .. s - 1 may land
//   while a probe runs, in any order: any snapshot between delta(<= s - kLag) and delta(<= s - 1)
//   gives a position between the two sets' M, and the later requests' common prefixes make it exact.
// Every cross-block wait is bounded (GreedySync::wait_ns, 1 s unless the caller set another limit);
// on expiry the waiter records PS_ERR_TIMEOUT and stops waiting, so the launch always ends.
//
// Caches that are not prefix-closed took a kernel of their own before: one block that walked delta and
// main 32 blocks a step on every instance whose hit rose, 50 us a decision (100 x 300: 15.2 ms of greedy
// pass, 0.46 here).

constexpr uint32_t kPipeThreads = 608;  // threads of every block of the launch
constexpr uint32_t kFeedRing = 8;       // rows staged in the deciding block's shared memory
constexpr unsigned long long kJobValid = 1ull << 63;  // a published job word (0 = not yet published)

// Bounded spin until *flag != 0 (acquire).  false after limit_ns (and the error bit is set).
__device__ __forceinline__ bool wait_flag(const uint32_t* flag, uint32_t* err, uint64_t limit_ns) {
  if (psk::ld_acquire_u32(flag) != 0u) return true;
  const uint64_t t0 = psk::globaltimer_ns();
  while (psk::ld_acquire_u32(flag) == 0u) {
    if (psk::globaltimer_ns() - t0 > limit_ns) {
      atomicOr(err, psk::kErrTimeout);
      return false;
    }
    __nanosleep(32);
  }
  return true;
}

// Bounded spin until *count >= want (acquire).  false after limit_ns (and the error bit is set).
__device__ __forceinline__ bool wait_count(const uint32_t* count, uint32_t want, uint32_t* err, uint64_t limit_ns) {
  if (psk::ld_acquire_u32(count) >= want) return true;
  const uint64_t t0 = psk::globaltimer_ns();
  while (psk::ld_acquire_u32(count) < want) {
    if (psk::globaltimer_ns() - t0 > limit_ns) {
      atomicOr(err, psk::kErrTimeout);
      return false;
    }
    __nanosleep(32);
  }
  return true;
}

// Bounded wait for a published job word; 0 after limit_ns (and the error bit is set).
__device__ __forceinline__ unsigned long long wait_job(const unsigned long long* job, uint32_t* err,
                                                       uint64_t limit_ns) {
  unsigned long long v = psk::ld_relaxed_u64(job);
  if (v & kJobValid) return v;
  const uint64_t t0 = psk::globaltimer_ns();
  for (;;) {
    v = psk::ld_relaxed_u64(job);
    if (v & kJobValid) return v;
    if (psk::globaltimer_ns() - t0 > limit_ns) {
      atomicOr(err, psk::kErrTimeout);
      return 0ull;
    }
    __nanosleep(32);
  }
}

__device__ __forceinline__ uint32_t job_pick(unsigned long long jb) { return (uint32_t)jb; }
__device__ __forceinline__ uint32_t job_hit(unsigned long long jb) { return (uint32_t)(jb >> 32) & 0x7FFFFFFFu; }

// Insert blocks, in groups of kInsertGroup: group g inserts the chain tails of jobs g, g + the number
// of groups, ...; the group's members split a tail by position (member m takes positions
// h + m * 256 + t, stride kInsertGroup * 256) and each adds 1 to the job's done count once its
// inserts are in, so the job's blocks are all in when the count reaches kInsertGroup.  A thread
// claims the home slots of kInsertBatch keys at once (the claims are independent) and follows the
// rare occupied home slot on its own.
using psgrid::kInsertGroup;
constexpr int kInsertBatch = 4;

// The committed tables, for caches that are not prefix-closed.
struct MainTables {
  const uint64_t* slots;
  const uint64_t* ovf;
  const psk::TableDesc* tdesc;
};

// First position in [from, nb) of a chain that instance i's committed table does not hold (a warp).
__device__ __noinline__ uint64_t main_first_miss(const MainTables& mt, uint32_t i, const uint64_t* chain, uint64_t from,
                                                 uint64_t nb) {
  const psk::TableDesc d = mt.tdesc[i];
  return psk::warp_first_miss_linear(
      from, nb, [&](uint64_t k) { return psk::main_contains(mt.slots, mt.ovf, d, __ldg(chain + k)); });
}

template <bool LIN>
__device__ __forceinline__ void insert_tail(psk::DeltaSlot* delta, uint64_t nslots, uint32_t j,
                                            const uint64_t* __restrict__ chain, uint64_t first, uint64_t nb,
                                            uint64_t stride, uint32_t* err) {
  for (uint64_t p0 = first; p0 < nb; p0 += kInsertBatch * stride) {
    uint64_t key[kInsertBatch], slot[kInsertBatch];
    unsigned long long old[kInsertBatch];
#pragma unroll
    for (int q = 0; q < kInsertBatch; ++q) {
      const uint64_t p = p0 + (uint64_t)q * stride;
      key[q] = p < nb ? __ldg(chain + p) : psk::kEmpty;
    }
#pragma unroll
    for (int q = 0; q < kInsertBatch; ++q) {
      old[q] = ~0ull;
      if (key[q] != psk::kEmpty && key[q] != psk::kTomb) {
        slot[q] = psk::delta_home(key[q], j, nslots);
        old[q] = atomicCAS(&delta[slot[q]].hash, psk::kEmpty, (unsigned long long)key[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < kInsertBatch; ++q) {
      if (key[q] == psk::kEmpty || key[q] == psk::kTomb) continue;
      if (old[q] == psk::kEmpty) {
        __stcg(&delta[slot[q]].tag, j + 1);
      } else if (LIN && psk::delta_contains_from(delta, nslots, j, key[q], slot[q])) {
        // another request of the window with this prefix brought the block to the instance before
      } else if (!psk::delta_insert_from(delta, nslots, j, key[q], psk::delta_next(slot[q], nslots))) {
        atomicOr(err, psk::kErrDeltaFull);
      }
    }
  }
}

template <bool LIN>
__device__ void insert_blocks(const psk::RowPre* __restrict__ rows, const uint64_t* __restrict__ hash, uint32_t R,
                              psk::DeltaSlot* delta, uint64_t nslots, uint32_t* err, const psk::GreedySync& sync,
                              uint32_t ib, uint32_t ninsert) {
  __shared__ unsigned long long s_job;
  const uint32_t t = threadIdx.x;
  const uint32_t group = ib / kInsertGroup, member = ib % kInsertGroup;
  const uint32_t groups = ninsert / kInsertGroup;
  for (uint32_t job = group; job < R; job += groups) {
    if (t == 0) s_job = wait_job(sync.jobs + job, err, sync.wait_ns);
    __syncthreads();
    const unsigned long long jb = s_job;
    if (jb == 0ull) return;  // block-uniform: timed out
    const uint32_t j = job_pick(jb);
    const uint32_t hj = job_hit(jb);
    // rows >= job + kLag are the only ones that read this job's inserts
    if (j != 0xFFFFFFFFu && job + psk::kLag < R) {
      const uint64_t off = __ldg(&rows[job].off);
      const uint32_t nb = __ldg(&rows[job].nb);
      insert_tail<LIN>(delta, nslots, j, hash + off, (LIN ? 0u : (uint64_t)hj) + member * blockDim.x + t, nb,
                       (uint64_t)kInsertGroup * blockDim.x, err);
    }
    __syncthreads();
    if (t == 0) {
      __threadfence();  // every thread's inserts before the count
      atomicAdd(sync.done + job, 1u);
    }
  }
}

// Probe blocks: block p probes rows p, p + their number, ... in order (see the section comment).
// Per row, everything that does not need the window's inserts comes first: replaying the published
// jobs <= s - kLag (which instances have window inserts, their last chain end, the picks of the
// row's ancestors), the hit0 row, the probe positions and the chain blocks there.  Only then does the
// block wait until those jobs' inserts are done, so after the wait one delta lookup per instance
// (and, rarely, a warp search) is left before the row is released.
template <int IPT, bool LIN>
__device__ void probe_rows(const psk::RowPre* __restrict__ rows, const uint64_t* __restrict__ hash, uint32_t R,
                           uint32_t I, const uint32_t* __restrict__ hit0, const float* __restrict__ tpf0,
                           const psk::DevModel& m, const psk::DeltaSlot* delta, uint64_t nslots, uint32_t* err,
                           const psk::GreedySync& sync, unsigned long long* smem_raw, uint32_t pb, uint32_t nprobe,
                           const MainTables& mt) {
  uint32_t* s_end = reinterpret_cast<uint32_t*>(smem_raw);  // chain end of the last job with blocks on i (0 = none)
  uint32_t* s_res = s_end + I;                               // search start / result per instance
  uint32_t* s_walk = s_res + I;                              // instances handed to a warp search
  __shared__ uint32_t s_nwalk;
  __shared__ int32_t s_ja[3];       // picks of the row's ancestors old enough to count (-1: none)
  __shared__ uint32_t s_jnb[3];     // their chain lengths
  __shared__ uint32_t s_replayed;   // jobs [0, s_replayed) are published and replayed
  __shared__ uint32_t s_done;       // jobs [0, s_done) have their inserts in the delta table
  __shared__ int s_abort;
  const uint32_t t = threadIdx.x;
  const uint32_t NT = blockDim.x;
  const int lane = t & 31, warp = t >> 5, NW = NT >> 5;
  unsigned long long cyc_done = 0;  // thread 0: cycles spent waiting for inserts
  for (uint32_t i = t; i < I; i += NT) s_end[i] = 0u;
  if (t == 0) {
    s_replayed = 0;
    s_done = 0;
    s_nwalk = 0;
    s_abort = 0;
  }
  __syncthreads();
  for (uint32_t s = pb; s < R; s += nprobe) {
    const uint64_t off = __ldg(&rows[s].off);
    const uint32_t nb = __ldg(&rows[s].nb);
    const uint32_t L = __ldg(&rows[s].L);
    const int64_t need = (int64_t)s - psk::kLag + 1;  // jobs [0, need) count for this row
    if (warp == 0) {
      // Replay the published jobs [replayed, need), 32 at a time; for each instance the latest of
      // them that has blocks sets its chain end.
      uint32_t f = s_replayed;
      bool abort = false;
      while ((int64_t)f < need && !abort) {
        const uint32_t x = f + (uint32_t)lane;
        const bool mine = (int64_t)x < need;
        unsigned long long jb = 0ull;
        if (mine) jb = wait_job(sync.jobs + x, err, sync.wait_ns);
        abort = __any_sync(0xffffffffu, mine && jb == 0ull);
        if (abort) break;
        const uint32_t nbx = mine ? __ldg(&rows[x].nb) : 0u;
        const uint32_t j = nbx ? job_pick(jb) : 0xFFFFFFFFu;  // (a prompt without a block inserts nothing)
        const unsigned same = __match_any_sync(0xffffffffu, j);
        if (j < I && (31 - __clz(same)) == lane) s_end[j] = nbx;
        const uint32_t n = (int64_t)f + 32 <= need ? 32u : (uint32_t)(need - (int64_t)f);
        f += n;
      }
      if (lane == 0) {
        s_replayed = f;
        s_abort = abort ? 1 : 0;
        const int32_t a[3] = {__ldg(&rows[s].par), __ldg(&rows[s].anc[0]), __ldg(&rows[s].anc[1])};
        const uint32_t anb[3] = {__ldg(&rows[s].par_nb), __ldg(&rows[s].anc_nb[0]), __ldg(&rows[s].anc_nb[1])};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          s_ja[q] = -1;
          s_jnb[q] = anb[q];
          if (!abort && a[q] >= 0 && (int64_t)a[q] < need) {
            const uint32_t j = job_pick(psk::ld_relaxed_u64(sync.jobs + a[q]));
            if (j < I) s_ja[q] = (int32_t)j;
          }
        }
      }
    }
    __syncthreads();
    if (s_abort) return;  // block-uniform
    const int32_t ja0 = s_ja[0], ja1 = s_ja[1], ja2 = s_ja[2];
    const uint32_t jn0 = s_jnb[0], jn1 = s_jnb[1], jn2 = s_jnb[2];
    uint32_t h0[IPT], pos[IPT];
    float tp0[IPT];
    uint64_t key[IPT];
    bool probe[IPT], walk[IPT];
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
      const uint32_t i = t + k * NT;
      probe[k] = false;
      walk[k] = false;
      if (i < I) {
        h0[k] = __ldg(hit0 + (uint64_t)s * I + i);
        tp0[k] = __ldg(tpf0 + (uint64_t)s * I + i);
        uint32_t p = h0[k];
        if ((int32_t)i == ja0 && jn0 > p) p = jn0;
        if ((int32_t)i == ja1 && jn1 > p) p = jn1;
        if ((int32_t)i == ja2 && jn2 > p) p = jn2;
        pos[k] = p;
        // s_end[i] != 0: the instance has window inserts visible to this row
        probe[k] = s_end[i] != 0u && p < nb;
        key[k] = probe[k] ? __ldg(hash + off + p) : 0ull;
      }
    }
    if (warp == 0) {
      // Wait until the inserts of jobs [done, need) are in: the leading run of done flags among the
      // next 32 is taken, and the first one not yet done is waited for.
      const long long c0 = clock64();
      uint32_t f = s_done;
      bool abort = false;
      while ((int64_t)f < need && !abort) {
        const uint32_t x = f + (uint32_t)lane;
        const bool ok = (int64_t)x < need && psk::ld_acquire_u32(sync.done + x) >= kInsertGroup;
        const unsigned okm = __ballot_sync(0xffffffffu, ok);
        const uint32_t nok = (okm == 0xffffffffu) ? 32u : (uint32_t)(__ffs(~okm) - 1);
        if (nok == 0u) {
          bool got = true;
          if (lane == 0) got = wait_count(sync.done + f, kInsertGroup, err, sync.wait_ns);
          abort = !__shfl_sync(0xffffffffu, got, 0);
          continue;
        }
        f += nok;
      }
      if (lane == 0) {
        s_done = f;
        s_abort = abort ? 1 : 0;
        cyc_done += (unsigned long long)(clock64() - c0);
      }
    }
    __syncthreads();
    if (s_abort) return;  // block-uniform
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
      const uint32_t i = t + k * NT;
      if ((probe[k] && psk::delta_contains(delta, nslots, i, key[k])) || (LIN && i < I && pos[k] > h0[k])) {
        walk[k] = true;
        s_res[i] = pos[k];
        s_walk[atomicAdd(&s_nwalk, 1u)] = i;
      }
    }
    __syncthreads();
    const uint32_t nwalk = s_nwalk;
    if (nwalk) {
      for (uint32_t x = warp; x < nwalk; x += NW) {
        const uint32_t i = s_walk[x];
        auto cached = [&](uint64_t k) { return k < nb && psk::delta_contains(delta, nslots, i, __ldg(hash + off + k)); };
        uint64_t hnew;
        if (!LIN) {
          hnew = psk::warp_first_miss_search_hint((uint64_t)s_res[i] + 1, nb, s_end[i], cached);
        } else {
          const uint64_t from = s_res[i], lim = __ldg(&rows[s].limit);
          hnew = from < lim ? psk::warp_first_miss_search_hint(from, lim, s_end[i], cached) : lim;
          hnew = main_first_miss(mt, i, hash + off, hnew, nb);
        }
        __syncwarp();
        if (lane == 0) s_res[i] = (uint32_t)hnew;
      }
      __syncthreads();
    }
    const uint32_t slot = s % psk::kHitSlots;
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
      const uint32_t i = t + k * NT;
      if (i < I) {
        const uint32_t h = walk[k] ? s_res[i] : pos[k];
        sync.hitring[(uint64_t)slot * sync.ring_stride + i] = h;
        sync.tpfring[(uint64_t)slot * sync.ring_stride + i] = h == h0[k] ? tp0[k] : psk::t_pf32(m, L, h);
      }
    }
    __syncthreads();
    if (t == 0) {
      s_nwalk = 0;
      __threadfence();  // the row's hits before its flag
      psk::st_release_u32(sync.ready + s, 1u);
    }
  }
  if (t == 0 && sync.stats) atomicAdd(sync.stats + psk::kGsProbeDoneWait, cyc_done);
}

// q and S within [0, 2^30): with L, n < 2^30 the sums S + L and q + n are exact in 32 bits.
__device__ __forceinline__ bool narrow_qs(int64_t q, int64_t S) {
  return q >= 0 && q < (1ll << 30) && S >= 0 && S < (1ll << 30);
}

// ---- deciding block -----------------------------------------------------------------------------
//
// Every decision evaluates its whole row on the current state; nothing about a row is known before
// the decision it follows, except the probed hits.  The block has up to kComputeWarps compute warps,
// a feeder warp, a hit warp and a publishing warp:
//   * compute thread t owns the instances IPT t .. IPT t + IPT - 1 and keeps their request-independent
//     terms (room, q, S, B, dec0, EMA factor, queueing TTFT, key bits) in registers for the whole
//     launch.  A pair needs its staged hit and T_pf and no other memory.  Per row: W, capacity,
//     latencies and key of every pair; W_min over the block (one warp reduction, one barrier); the
//     recompute filter; the smallest (key, tie) of each warp into shared memory; the step's barrier,
//     after which every warp combines the warps' minima by itself.
//   * the feeder copies each row's constants, probed hits and T_pf into a ring in shared memory.
//   * the hit warp raises row s + 1's hits, while row s is decided, on the instances that took requests
//     s - kLcpBack + 1 .. s - 1, to the common chain prefix with them (lane k holds the pick of request
//     s - 1 - k); the pick of s itself is raised by its owner one step later.
//   * the publishing warp hands decision s - 1 to the insert and probe blocks and writes the outputs.
// A step is a chain of latencies: barrier, the last decision (two warp votes), its owner's one-pair
// update, W_min (reduction, barrier, reduction), the warp's pick (reduction, vote).  Measured per
// decision, before -> now (before: row summaries computed by other blocks 8 decisions ahead and
// corrected by one warp, with helper warps; 1.25 us of helper phase a step, and a pass over the row by
// one warp, 20 to 30 us, where the summary did not cover the pick):
//   64 instances 1.22 -> 0.53 us, 201: 1.43 -> 0.67, 256: 1.41 -> 0.65, 999: 3.3 -> 0.85, 1024: 1.60 -> 0.82.
// 1024 instances are bound by issue slots (about 215 instructions a warp and step on 16 warps, 55% of the
// slots) beside the chain, small pools by the chain.  The pick's owner takes its place in the row by two
// blocks, its W before the rest (1024 x 16384: 14.4 ms, 14.7 in one), and a warp's pick is handed on by
// the lane that finds itself the only one, before the vote that says so (15.2 ms if after it).

constexpr uint32_t kComputeWarps = 16;
constexpr uint32_t kFeederWarp = kComputeWarps;
constexpr uint32_t kHitWarp = kComputeWarps + 1;
constexpr uint32_t kPublishWarp = kComputeWarps + 2;
static_assert(kPipeThreads == 32 * (kComputeWarps + 3), "compute warps, the feeder, the hit warp, the publisher");
static_assert(psk::kLcpBack == 32, "one lane of the hit warp per recent request");

// Instance state of the deciding block in shared memory, [Ip] each, 8-byte arrays first: the truth
// behind the owners' registers (36 bytes per instance).
struct InstSmem {
  int64_t* q;
  int64_t* S;
  int64_t* M;
  int32_t* b;
  int32_t* qr;
  int32_t* Bmax;
  int32_t* pad;
  // with 32-bit sums: {q, S, KV room (-1: no decode slot), slots left} and {key low (qr), key high (b), B, -}
  // per instance, over the same memory
  int4* qs;
  uint4* kb;
};
constexpr size_t kInstSmemBytes = 3 * sizeof(int64_t) + 4 * sizeof(int32_t);
static_assert(kInstSmemBytes >= sizeof(int4) + sizeof(uint4), "both forms fit");

__device__ __forceinline__ InstSmem inst_smem(unsigned long long* raw, uint32_t Ip) {
  InstSmem a;
  a.q = reinterpret_cast<int64_t*>(raw);
  a.S = a.q + Ip;
  a.M = a.S + Ip;
  a.b = reinterpret_cast<int32_t*>(a.M + Ip);
  a.qr = a.b + Ip;
  a.Bmax = a.qr + Ip;
  a.pad = a.Bmax + Ip;
  a.qs = reinterpret_cast<int4*>(raw);
  a.kb = reinterpret_cast<uint4*>(a.qs + Ip);
  return a;
}

// IPT consecutive 32-bit words of shared memory (aligned to IPT words, at most 4 per load).
template <int IPT>
__device__ __forceinline__ void lds_words(const uint32_t* p, uint32_t (&v)[IPT]) {
  if constexpr (IPT == 1) {
    v[0] = p[0];
  } else if constexpr (IPT == 2) {
    const uint2 x = *reinterpret_cast<const uint2*>(p);
    v[0] = x.x;
    v[1] = x.y;
  } else {
#pragma unroll
    for (int k = 0; k < IPT; k += 4) {
      const uint4 x = *reinterpret_cast<const uint4*>(p + k);
      v[k] = x.x;
      v[k + 1] = x.y;
      v[k + 2] = x.z;
      v[k + 3] = x.w;
    }
  }
}

// A packed key's rank: a 32-bit word whose unsigned order never contradicts the keys' (equal ranks
// need the full comparison), so one warp reduction nearly always finds the smallest key.  Class 0:
// the key's upper 31 bits; class 1: the value as fp32 rounded towards zero, above every class-0 rank;
// no key: all ones.
__device__ __forceinline__ uint32_t key_rank(uint64_t key) {
  const uint32_t c0 = (uint32_t)(key >> 31);
  const uint32_t c1 = 0x80000000u | __float_as_uint(__ull2float_rz(key & ((1ull << 62) - 1)));
  return key == psk::kNoKey ? 0xFFFFFFFFu : ((key >> 62) ? c1 : c0);
}

// The rank and the packed key of a pair from 32-bit words of its state, in every instance order (GEN; else
// Algorithm 1's).  With a 64-bit key by the order for every pair and branches on the order, the other orders cost
// 90 instructions a pair more: 1025 instances (four a thread) took 1.91 us a decision in the D order, 1.83 in
// H-C-Q and 2.00 with Eq. 9; 1.52, 1.43 and 1.49 now (Algorithm 1's order, whose kernels have their rank
// written out: 1.11).  Ranks are made for every pair, keys only where ranks are equal, from two words of the pair:
// {D-C-Q key bits of qr, of b} in T (H-C-Q: the headroom's bits) and under the D-C-Q fallback, {q + n, B}
// under the product.
// Where qr comes last in an order, the tie word of a pair in T starts with it, so that nearly always equal ranks
// in T mean that the smallest tie word wins (exact).
struct PairOrder {  // masks of the launch's order: a step has no branch on it
  uint32_t d_mask, c_mask, q_mask;  // what a rank in T takes: b, cached blocks, queued requests ...
  uint32_t head_mask, head_shift;   // ... or (H-C-Q) the headroom, and its bits that the rank leaves out
  uint32_t fb_mask;                 // D-C-Q fallback
  bool head_all;                    // head_mask is set
  uint32_t tie_q;                   // the part of the tie word above the instance
  uint32_t ex_mask, ex_any;         // a rank in T leaves only the tie word to compare if (rank & ex_mask) | ex_any
  __device__ __forceinline__ bool exact(uint32_t rank) const {
    return rank < 0x80000000u && ((rank & ex_mask) | ex_any) != 0u;
  }
  // In T: b, then up to 13 bits of h (more is better) or of qr; H-C-Q: the headroom (head: f2ord of it).
  __device__ __forceinline__ uint32_t in_t(uint32_t kq, uint32_t kdh, uint32_t h, uint32_t head) const {
    return ((kdh << 1) & d_mask) | ((8191u - min(h, 8191u)) & c_mask) | ((kq >> 5) & q_mask) |
           ((head >> head_shift) & head_mask);
  }
  // In C \ T: the product rounded towards zero as fp32 (p), or the D-C-Q order's bits.
  __device__ __forceinline__ uint32_t fallback(uint32_t kdh, uint32_t h, float p) const {
    const uint32_t dc = (kdh << 1) | (8191u - min(h, 8191u));
    return 0x80000000u | ((dc >> 1) & fb_mask) | (__float_as_uint(p) & ~fb_mask);
  }
};

__device__ __forceinline__ PairOrder pair_order(const psk::DevModel& m) {
  const bool dc = m.sel == psk::kSelDCQ || m.sel == psk::kSelDC, dq = m.sel == psk::kSelDQ, hcq = m.sel == psk::kSelHCQ;
  PairOrder o;
  o.d_mask = hcq ? 0u : ~0u;
  o.c_mask = dc ? 8191u : 0u;
  o.q_mask = m.sel == psk::kSelDQC ? 8191u : 0u;
  o.head_mask = hcq ? 0x7FFFFFFFu : 0u;
  o.head_all = hcq;
  o.fb_mask = m.fb_dcq ? 0x7FFFFFFFu : 0u;
  o.tie_q = m.sel == psk::kSelDCQ || dq || hcq ? 0x3FFFFu : 0u;
  o.ex_mask = dc ? 8191u : 0u;  // 0 there: 8191 blocks or more, which the rank does not tell apart
  o.ex_any = dq || m.sel == psk::kSelD ? 1u : 0u;
  o.head_shift = m.slo_off ? 5u : 0u;  // an admitted pair's headroom is positive, unless everything is admitted
  return o;
}

template <bool GEN>
__device__ __forceinline__ uint64_t pair_key(const psk::DevModel& m, uint32_t rank, uint2 w, uint32_t h) {
  if (rank == 0xFFFFFFFFu) return psk::kNoKey;
  const uint64_t kd = ((uint64_t)w.y << 32) | w.x;
  const uint64_t C = (1u << 26) - 1u - h;
  if (rank & 0x80000000u)
    return psk::packed_key(1u, GEN && m.fb_dcq ? kd | (C << 18) : (uint64_t)w.x * (uint64_t)w.y);
  if (!GEN) return kd | (C << 18);
  return m.sel == psk::kSelHCQ ? ((uint64_t)w.x << 26) | C : psk::key0_from_dcq(m, kd) | psk::hit_bits(m, h);
}

// The lane holding the warp's smallest (key, tie), -1 if no lane has a key; rank = key_rank(key).
__device__ __forceinline__ int warp_argmin(uint32_t rank, uint64_t key, uint32_t tie) {
  const uint32_t mr = __reduce_min_sync(0xffffffffu, rank);
  unsigned who = __ballot_sync(0xffffffffu, rank == mr);
  if (mr == 0xFFFFFFFFu) return -1;
  if (who & (who - 1u)) {  // equal ranks: compare the keys, then the tie words (warp-uniform)
    bool in = rank == mr;
    const uint32_t mhi = __reduce_min_sync(0xffffffffu, in ? (uint32_t)(key >> 32) : 0xFFFFFFFFu);
    in = in && (uint32_t)(key >> 32) == mhi;
    const uint32_t mlo = __reduce_min_sync(0xffffffffu, in ? (uint32_t)key : 0xFFFFFFFFu);
    in = in && (uint32_t)key == mlo;
    const uint32_t mt = __reduce_min_sync(0xffffffffu, in ? tie : 0xFFFFFFFFu);
    who = __ballot_sync(0xffffffffu, in && tie == mt);  // tie words are unique
  }
  return __ffs(who) - 1;
}

// What a step needs of a row's constants (RowPre's second word and a few more).
struct StepRow {
  float t_cached, c_max, ttft_max, tpot_lim, tpot_target;
  uint32_t L;
};

__device__ __forceinline__ StepRow step_row(const psk::RowPre& x) {
  const float4 w1 = reinterpret_cast<const float4*>(&x)[1];
  StepRow r;
  r.L = x.L;
  r.t_cached = w1.x;
  r.c_max = w1.y;
  r.tpot_lim = w1.z;
  r.ttft_max = w1.w;
  r.tpot_target = x.tpot_target;
  return r;
}

using psk::wait_smem_at_least;

template <int IPT, bool GEN, bool EQ9, bool LIN>
__device__ void decide_rows(const psk::RowPre* __restrict__ rows, uint32_t R, uint32_t I, psk::StateSoA committed,
                            psk::StateSoA pending, const psk::DevModel& m, int32_t* assign, uint8_t* __restrict__ path,
                            uint32_t* __restrict__ hit_chosen, uint32_t* err, const psk::GreedySync& sync,
                            unsigned long long* smem_raw, const uint64_t* __restrict__ hash, const MainTables& mt,
                            uint64_t tokens) {
  const uint32_t Ip = sync.ring_stride;
  const InstSmem a = inst_smem(smem_raw, Ip);
  uint32_t* s_hitr = reinterpret_cast<uint32_t*>(a.pad + Ip);  // [kFeedRing][Ip] hits
  uint32_t* s_tpfr = s_hitr + kFeedRing * Ip;                   // [kFeedRing][Ip] T_pf at them (bits)
  __shared__ psk::RowPre s_row[kFeedRing];
  __shared__ uint32_t s_rank[2][kComputeWarps];            // a step's warp minima: their ranks (all ones: none) ...
  __shared__ uint2 s_th[2][kComputeWarps];                 // ... tie word and hit ...
  __shared__ uint2 s_key[2][kComputeWarps];                // ... and packed key, or pair_key's words (narrow)
  __shared__ uint32_t s_w[kComputeWarps];                  // a step's warp minima of W over A (f2ord)
  __shared__ uint32_t s_begun;                             // steps [0, s_begun) have begun
  __shared__ uint32_t s_landed;                            // rows [0, s_landed) are staged
  __shared__ volatile int s_fail;                          // a bounded wait ran out (feeder and hit warp)
  // The step whose barrier is the last one, once a wait has run out (the hit warp sets it before it arrives
  // there).  A step number, not a flag: a warp that looks late at step s must not leave for step s + 1.
  __shared__ volatile uint32_t s_stop;
  const uint32_t t = threadIdx.x;
  const int lane = (int)(t & 31u);
  const uint32_t warp = t >> 5;
  const uint32_t ncw = (I + 32u * IPT - 1) / (32u * IPT);  // compute warps in use
  if (t < kComputeWarps) {
    s_w[t] = 0xFFFFFFFFu;
  }
  // An instance only takes requests that fit its KV room, so S stays below max(S, M), it gains no more than the
  // window's tokens, and q gains at most what S gains: with these bounds 32 bits hold every q and S of the
  // window.  (A KV room above 2^31 - 1 counts as that much, still more than any prompt at the end.)
  bool narrow = true;
  for (uint32_t i = t; i < I; i += kPipeThreads) {
    const int64_t M = committed.M[i], S = committed.S[i], q = committed.q[i];
    const int64_t gain = M > S ? (M - S < (int64_t)tokens ? M - S : (int64_t)tokens) : 0;
    narrow = narrow && S + gain < (1ll << 30) && q + gain < (1ll << 30);
  }
  if (t == 0) {
    s_begun = 0u;
    s_landed = 0u;
    s_fail = 0;
    s_stop = 0xFFFFFFFFu;
  }
  narrow = __syncthreads_and(narrow ? 1 : 0) != 0;
  if (!narrow) {
    for (uint32_t i = t; i < I; i += kPipeThreads) {
      a.b[i] = committed.b[i];
      a.qr[i] = committed.qr[i];
      a.q[i] = committed.q[i];
      a.S[i] = committed.S[i];
      a.M[i] = committed.M[i];
      a.Bmax[i] = committed.Bmax[i];
    }
    __syncthreads();
  }
  if (warp >= ncw && warp < kComputeWarps) return;
  const uint32_t nall = 32u * (ncw + 2u), ncmp = 32u * ncw;
  auto bar_step = [&]() { asm volatile("bar.sync 2, %0;" ::"r"(nall) : "memory"); };     // compute, hit and publishing warps
  auto bar_compute = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(ncmp) : "memory"); };  // compute warps
  // Step x's pick from the warps' minima (after the next step's barrier), in every lane: the warp that
  // holds it, -1 if rejected.  r: this lane's entry of s_rank[x & 1] (all ones past the warps in use).
  auto key_at = [&](uint32_t x, uint32_t r, uint32_t l) {
    const uint2 w = s_key[x & 1u][l];
    return narrow ? pair_key<GEN>(m, r, w, s_th[x & 1u][l].y) : ((uint64_t)w.y << 32) | w.x;
  };
  const PairOrder order = pair_order(m);
  auto exact = [&](uint32_t r) { return GEN && narrow && order.exact(r); };
  auto decision = [&](uint32_t x, uint32_t r) {
    const uint32_t mr = __reduce_min_sync(0xffffffffu, r);
    const unsigned who = __ballot_sync(0xffffffffu, r == mr);
    int src = __ffs(who) - 1;
    if (who & (who - 1u)) {  // equal ranks (or nobody has a pair)
      const uint32_t l = (uint32_t)lane < ncw ? lane : 0u;
      const uint32_t tie = s_th[x & 1u][l].x;
      if (exact(mr)) {
        const uint32_t mt = __reduce_min_sync(0xffffffffu, r == mr ? tie : 0xFFFFFFFFu);
        src = __ffs(__ballot_sync(0xffffffffu, r == mr && tie == mt)) - 1;
      } else {
        src = warp_argmin(r, key_at(x, r, l), tie);
      }
    }
    return src;
  };
  auto rank_of = [&](uint32_t x) { return (uint32_t)lane < ncw ? s_rank[x & 1u][lane] : 0xFFFFFFFFu; };

  // LIN: what the last pick's hit on this row rises to (0: it does not), called by its owner's warp.
  auto extend = [&](const psk::RowPre& row, uint32_t j, uint32_t hj) {
    const uint32_t l = min(row.lcp[0], row.limit);
    return l > hj ? (uint32_t)main_first_miss(mt, j, hash + row.off, l, row.nb) : 0u;
  };

  if (warp == kFeederWarp) {
    // Rows are staged as soon as they are probed, several at once when they are ready together (so the
    // round trips to L2 are shared).  Step s reads row s (and the length of row s - 1), the hit warp
    // row s + 1 in the meantime: once step s has begun, rows up to s + kFeedRing - 2 may be staged.
    unsigned long long cyc_slot = 0, cyc_ready = 0;
    for (uint32_t x = 0; x < R;) {
      uint32_t n = 0;
      const long long cs = clock64();
      if (lane == 0 &&
          (x + 3 <= kFeedRing || wait_smem_at_least(&s_begun, x + 3 - kFeedRing, &s_fail, err, sync.wait_ns))) {
        cyc_slot += (unsigned long long)(clock64() - cs);
        n = psk::ld_relaxed_cta_shared_u32(&s_begun) + kFeedRing - 2 - x;
        psk::fence_acq_rel_cta();
        const long long c0 = clock64();
        if (!wait_flag(sync.ready + x, err, sync.wait_ns)) n = 0;
        cyc_ready += (unsigned long long)(clock64() - c0);
      }
      n = __shfl_sync(0xffffffffu, n, 0);
      if (n == 0) {  // warp-uniform: a wait ran out
        if (lane == 0) s_fail = 1;
        break;
      }
      n = min(n, R - x);
      const bool rdy = (uint32_t)lane < n && psk::ld_acquire_u32(sync.ready + x + lane) != 0u;
      const unsigned rm = __ballot_sync(0xffffffffu, rdy) | 1u;  // row x is ready
      n = (uint32_t)(__ffs(~rm) - 1);
      for (uint32_t y = x; y < x + n; ++y) {
        const uint32_t slot = y % kFeedRing;
        if (lane < psk::kRowWords)
          psk::cp_async16(reinterpret_cast<uint4*>(&s_row[slot]) + lane, reinterpret_cast<const uint4*>(rows + y) + lane);
        const uint4* src_h = reinterpret_cast<const uint4*>(sync.hitring + (uint64_t)(y % psk::kHitSlots) * Ip);
        const uint4* src_t = reinterpret_cast<const uint4*>(sync.tpfring + (uint64_t)(y % psk::kHitSlots) * Ip);
        uint4* dst_h = reinterpret_cast<uint4*>(s_hitr + slot * Ip);
        uint4* dst_t = reinterpret_cast<uint4*>(s_tpfr + slot * Ip);
        for (uint32_t w = (uint32_t)lane; w < Ip / 4; w += 32) {
          psk::cp_async16(dst_h + w, src_h + w);
          psk::cp_async16(dst_t + w, src_t + w);
        }
      }
      psk::cp_async_commit();
      psk::cp_async_wait_all();
      __syncwarp();
      x += n;
      if (lane == 0) psk::st_release_cta_shared_u32(&s_landed, x);
    }
    if (lane == 0 && sync.stats) {
      atomicAdd(sync.stats + psk::kGsFeedSlotWait, cyc_slot);
      atomicAdd(sync.stats + psk::kGsFeedWait, cyc_ready);
    }
    return;
  }

  if (warp == kHitWarp) {
    int32_t pk = -1;  // lane k: the pick of request s - 1 - k (-1: none or rejected)
    unsigned long long cyc_wait = 0;
    for (uint32_t s = 0; s <= R; ++s) {
      // rows s and s + 1 must be staged when step s begins
      const long long c0 = clock64();
      if (lane == 0 && !wait_smem_at_least(&s_landed, s + 2 < R ? s + 2 : R, &s_fail, err, sync.wait_ns)) s_stop = s;
      cyc_wait += (unsigned long long)(clock64() - c0);
      __syncwarp();
      bar_step();
      if (s_stop <= s) {
        if (lane == 0) s_fail = 1;  // the feeder stops too
        break;
      }
      if (lane == 0) psk::st_release_cta_shared_u32(&s_begun, s + 1);
      if (s > 0) {
        const int src = decision(s - 1, rank_of(s - 1));
        pk = __shfl_up_sync(0xffffffffu, pk, 1);
        if (lane == 0) pk = src < 0 ? -1 : (int32_t)(s_th[(s - 1) & 1u][src].x & psk::kTieInstMask);
      }
      if (s + 1 < R) {  // request s - 1 - lane is lane + 2 places before row s + 1
        const uint32_t slot = (s + 1) % kFeedRing;
        const psk::RowPre& row = s_row[slot];
        const bool up = pk >= 0 && lane + 1 < psk::kLcpBack;
        uint32_t* hp = s_hitr + slot * Ip + (up ? pk : 0);
        bool rose = false;
        if (up) {
          const uint32_t l = LIN ? min(row.lcp[lane + 1], row.limit) : row.lcp[lane + 1];
          rose = atomicMax(hp, l) < l;
        }
        __syncwarp();
        if (LIN) {  // on from the common prefix in the committed table
          for (unsigned rm = __ballot_sync(0xffffffffu, rose); rm; rm &= rm - 1u) {
            const uint32_t i = (uint32_t)__shfl_sync(0xffffffffu, pk, __ffs(rm) - 1);
            const uint64_t hx = main_first_miss(mt, i, hash + row.off, s_hitr[slot * Ip + i], row.nb);
            __syncwarp();
            if (lane == 0) s_hitr[slot * Ip + i] = (uint32_t)hx;
            __syncwarp();
          }
        }
        if (rose) s_tpfr[slot * Ip + pk] = __float_as_uint(psk::t_pf32(m, row.L, *hp));
        __syncwarp();
      }
    }
    if (lane == 0 && sync.stats) atomicAdd(sync.stats + psk::kGsDecideWait, cyc_wait);
    return;
  }

  if (warp == kPublishWarp) {
    // Global stores stay in a warp of their own: a fence behind them would wait for their round trip.
    for (uint32_t s = 0; s <= R; ++s) {
      bar_step();
      if (s_stop <= s) break;
      if (s == 0) continue;
      const int src = decision(s - 1, rank_of(s - 1));
      uint2 th = make_uint2(0xFFFFFFFFu, 0u);
      uint32_t cls = 2u;
      if (src >= 0) {
        th = s_th[(s - 1) & 1u][src];
        cls = s_rank[(s - 1) & 1u][src] >> 31;
      }
      const uint32_t j = src < 0 ? 0xFFFFFFFFu : th.x & psk::kTieInstMask;
      if (lane == 0) psk::st_relaxed_u64(sync.jobs + s - 1, kJobValid | ((unsigned long long)th.y << 32) | j);
      if (lane == 1) assign[s - 1] = (int32_t)j;
      if (lane == 2) path[s - 1] = (uint8_t)cls;
      if (lane == 3) hit_chosen[s - 1] = th.y;
    }
    return;
  }

  const uint32_t i0 = t * IPT;
  const bool loads = i0 < Ip;  // rows are padded to Ip, a multiple of 8 (the padding's room is -1)
  const long long cyc0 = clock64();
  bool stopped = false;
  if (narrow) {
    // ---- compute warps --------------------------------------------------------------------------
    // Every q and S of the window stays in [0, 2^30): 32-bit state.  After the step's barrier the whole
    // row is evaluated on the state without the last decision, side by side with the chain that finds
    // that decision (the rank reductions); the pick's owner then replaces its one pair.
    int32_t room[IPT], q32[IPT], S32[IPT], Bp[IPT];
    float dec0[IPT], fe[IPT], tq[IPT];
    uint32_t kq[IPT], kdh[IPT];  // D-C-Q key bits of (b, qr): low (qr) and high (b) words
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
      const uint32_t i = i0 + (uint32_t)k;
      room[k] = -1;
      q32[k] = S32[k] = 0;
      Bp[k] = 1;
      dec0[k] = fe[k] = tq[k] = 0.0f;
      kq[k] = kdh[k] = 0u;
      if (i < I) {
        const int32_t b = committed.b[i], qr = committed.qr[i], Bmax = committed.Bmax[i];
        const int64_t q = committed.q[i], S = committed.S[i];
        const psk::InstTerms it = psk::inst_terms(m, b, qr, q, Bmax);
        const uint64_t kd = psk::dcq_key0(b, qr);
        room[k] = it.okB ? psk::kv_room(S, committed.M[i]) : -1;
        dec0[k] = it.dec0;
        fe[k] = it.f;
        tq[k] = it.tq;
        Bp[k] = it.Bp;
        kq[k] = (uint32_t)kd;
        kdh[k] = (uint32_t)(kd >> 32);
        q32[k] = (int32_t)q;
        S32[k] = (int32_t)S;
        a.qs[i] = make_int4(q32[k], S32[k], room[k], Bmax - it.Bp);
        a.kb[i] = make_uint4(kq[k], kdh[k], (uint32_t)Bp[k], 0u);
      }
    }
    const float den = m.lout > 1.0f ? m.lout : 1.0f;
    // One pair on the given state: W (+infinity outside A), and the rank and the tie word it has in C (and, under
    // H-C-Q, its headroom's bits).  Without branches, so that a thread's pairs overlap.
    auto pair = [&](const StepRow& rc, uint32_t i, uint32_t h, float tpf, int32_t rm, int32_t q, int32_t S, int32_t B,
                    float d0, float f, float tqv, uint32_t kql, uint32_t kh, float* W, uint32_t* head, uint32_t* rank,
                    uint32_t* tie) {
      const int32_t n = (int32_t)rc.L - (int32_t)(h << 4);
      *W = (int32_t)rc.L <= rm ? __fsub_rn(tpf, rc.t_cached) : INFINITY;
      float dec = __fadd_rn(d0, __fmul_rn(m.b2, __int2float_rn(S + (int32_t)rc.L)));
      dec = __fmul_rn(dec, f);
      const float qnf = __int2float_rn(q + n);
      // queued prefill, or Eq. 9's interference
      const float tpot = __fadd_rn(dec, EQ9 ? (B > 1 ? __fdiv_rn(tpf, den) : 0.0f) : __fmul_rn(m.g_q, qnf));
      const float ttft = __fadd_rn(tpf, tqv);
      const bool adm = (tpot < rc.tpot_lim) & (ttft <= rc.ttft_max);
      // The product rounded towards zero: both factors exact in fp32, else from the 64-bit product, the same
      // rounding of the same value.
      const uint64_t qn = (uint64_t)(uint32_t)(q + n);
      const uint64_t v1 = qn * (uint64_t)(uint32_t)B;
      const float p1 = (uint32_t)qn < (1u << 24) ? __fmul_rz(qnf, __int2float_rn(B)) : __ull2float_rz(v1);
      *tie = i;
      if constexpr (GEN) {
        *tie |= (kql & (adm ? order.tie_q : 0u)) << 12;
        *head = psk::f2ord(__fsub_rn(rc.tpot_target, tpot));
        *rank = adm ? order.in_t(kql, kh, h, *head) : order.fallback(kh, h, p1);
      } else {  // Algorithm 1's order: D and up to 13 bits of C in T, the product in C \ T
        *rank = adm ? (kh << 1) | (8191u - min(h, 8191u)) : 0x80000000u | __float_as_uint(p1);
      }
    };
    uint32_t Lprev = 0;  // length of request s - 1
    for (uint32_t s = 0;; ++s) {
      bar_step();
      // the last decision's ranks and picks, and this row (past the last row: any staged one)
      const uint32_t par = (s - 1) & 1u;
      const bool held = (uint32_t)lane < ncw && s > 0;
      const uint32_t er = held ? s_rank[par][lane] : 0xFFFFFFFFu;
      const uint2 eth = s_th[par][held ? lane : 0];
      const uint32_t slot = (s < R ? s : R - 1) % kFeedRing;
      const psk::RowPre& row = s_row[slot];
      const StepRow rc = step_row(row);
      const uint32_t l0 = row.lcp[0];
      uint32_t h[IPT], tb[IPT];
      if (loads) {
        lds_words<IPT>(s_hitr + slot * Ip + i0, h);
        lds_words<IPT>(s_tpfr + slot * Ip + i0, tb);
      } else {
#pragma unroll
        for (int k = 0; k < IPT; ++k) h[k] = tb[k] = 0u;
      }
      if (s_stop <= s) {
        stopped = true;
        break;
      }
      const uint32_t mr = __reduce_min_sync(0xffffffffu, er);
      uint32_t jt = __reduce_min_sync(0xffffffffu, er == mr ? eth.x : 0xFFFFFFFFu);
      uint32_t H = __reduce_min_sync(0xffffffffu, er == mr ? eth.y : 0xFFFFFFFFu);
      const unsigned who = __ballot_sync(0xffffffffu, er == mr);
      float W[IPT];
      uint32_t head[IPT], rank[IPT], tie[IPT];
#pragma unroll
      for (int k = 0; k < IPT; ++k)
        pair(rc, i0 + (uint32_t)k, h[k], __uint_as_float(tb[k]), room[k], q32[k], S32[k], Bp[k], dec0[k], fe[k], tq[k],
             kq[k], kdh[k], &W[k], &head[k], &rank[k], &tie[k]);
      bool own = false;  // this thread owns the last pick
      uint32_t j = 0, hj = 0;
      int4 x = make_int4(0, 0, 0, 0);
      float tpfj = 0.0f;
      if (mr != 0xFFFFFFFFu) {
        if (who & (who - 1u)) {  // equal ranks
          const int src = exact(mr) ? __ffs(__ballot_sync(0xffffffffu, er == mr && eth.x == jt)) - 1
                                    : warp_argmin(er, key_at(par, er, held ? lane : 0), eth.x);
          jt = __shfl_sync(0xffffffffu, eth.x, src);
          H = __shfl_sync(0xffffffffu, eth.y, src);
        }
        j = jt & psk::kTieInstMask;
        uint32_t lj = l0;
        if (LIN && j / (32u * IPT) == warp) lj = extend(row, j, s_hitr[slot * Ip + j]);
        if (j / IPT == t) {
          // its state takes request s - 1 (qr + 1, q + L - 16 H, S + L), and its hit rises to the common
          // prefix of the two requests: first its W, then (the second block) the rest
          own = true;
          x = a.qs[j];
          hj = s_hitr[slot * Ip + j];
          x.w -= 1;
          x.z = x.w < 0 ? -1 : x.z - (int32_t)Lprev;
          hj = lj > hj ? lj : hj;
          tpfj = psk::t_pf32(m, rc.L, hj);
          const float Wj = (int32_t)rc.L <= x.z ? __fsub_rn(tpfj, rc.t_cached) : INFINITY;
#pragma unroll
          for (int k = 0; k < IPT; ++k)
            if (i0 + (uint32_t)k == j) W[k] = Wj;
        }
      }
      if (own) {
        uint4 y = a.kb[j];
        x.x += (int32_t)Lprev - (int32_t)(H << 4);
        x.y += (int32_t)Lprev;
        y.x += 1u;
        y.z += 1u;
        a.qs[j] = x;
        a.kb[j] = y;
        const float d0 = __fadd_rn(m.b0, __fmul_rn(m.b1, __int2float_rn((int32_t)y.z)));
        const float f = psk::ema_factor(m, (int32_t)y.z);
        const float tqv =
            __fadd_rn(__fmul_rn(m.a0, __int2float_rn((int32_t)(y.x & 0x3FFFFu))), __fmul_rn(m.a1, __int2float_rn(x.x)));
        float Wj;
        uint32_t headj, rankj, tiej;
        pair(rc, j, hj, tpfj, x.z, x.x, x.y, (int32_t)y.z, d0, f, tqv, y.x, y.y, &Wj, &headj, &rankj, &tiej);
#pragma unroll
        for (int k = 0; k < IPT; ++k)
          if (i0 + (uint32_t)k == j) {
            if (GEN) head[k] = headj;
            rank[k] = rankj;
            tie[k] = tiej;
            h[k] = hj;
            q32[k] = x.x;
            S32[k] = x.y;
            room[k] = x.z;
            Bp[k] = (int32_t)y.z;
            kq[k] = y.x;
            dec0[k] = d0;
            fe[k] = f;
            tq[k] = tqv;
          }
      }
      float wbest = W[0];
#pragma unroll
      for (int k = 1; k < IPT; ++k) wbest = fminf(wbest, W[k]);
      uint32_t wmin_o = __reduce_min_sync(0xffffffffu, psk::f2ord(wbest));
      if (ncw > 1u && lane == 0) s_w[warp] = wmin_o;
      if (s == R) break;
      Lprev = rc.L;
      if (ncw > 1u) {
        bar_compute();
        wmin_o = __reduce_min_sync(0xffffffffu, s_w[lane & (kComputeWarps - 1)]);
      }
      const float wmin = psk::ord2f(wmin_o);
      // ranks after the recompute filter (a pair outside A has W = +infinity)
#pragma unroll
      for (int k = 0; k < IPT; ++k) rank[k] = __fsub_rn(W[k], wmin) <= rc.c_max ? rank[k] : 0xFFFFFFFFu;
      uint32_t rbest = rank[0];
#pragma unroll
      for (int k = 1; k < IPT; ++k) rbest = min(rbest, rank[k]);
      const uint32_t mw = __reduce_min_sync(0xffffffffu, rbest);
      uint32_t n_eq = 0;
      uint2 bk;
      uint32_t bt, bh;
      // The thread's smallest, picked beside the reduction.  Its key stays two words of the pair's state: only
      // equal ranks read it, and built for every pair it takes a tenth of a step's instructions (Algorithm 1's,
      // 1024 x 16384: 14.36 ms with it, 14.18 without).
      auto key_words = [&](int k) {
        const bool in_t = rank[k] < 0x80000000u;
        if constexpr (GEN) {
          const bool kd = in_t || order.fb_mask;
          const uint32_t x = order.head_all && in_t ? head[k] : kq[k];
          return make_uint2(kd ? x : (uint32_t)(q32[k] + ((int32_t)rc.L - (int32_t)(h[k] << 4))),
                            kd ? kdh[k] : (uint32_t)Bp[k]);
        } else {
          return make_uint2(in_t ? kq[k] : (uint32_t)(q32[k] + ((int32_t)rc.L - (int32_t)(h[k] << 4))),
                            in_t ? kdh[k] : (uint32_t)Bp[k]);
        }
      };
#pragma unroll
      for (int k = 0; k < IPT; ++k)
        if (k == 0 || rank[k] == rbest) {
          if (rank[k] == rbest) ++n_eq;
          bk = key_words(k);
          bt = tie[k];
          bh = h[k];
        }
      const bool has = rbest == mw;
      // the lane that holds it hands it on at once (with equal ranks several do, and the smallest again below)
      if (has) {
        s_rank[s & 1u][warp] = mw;
        s_th[s & 1u][warp] = make_uint2(bt, bh);
        s_key[s & 1u][warp] = bk;
      }
      const unsigned lanes = __ballot_sync(0xffffffffu, has);
      const unsigned many = IPT > 1 ? __ballot_sync(0xffffffffu, has && n_eq > 1u) : 0u;
      if (mw != 0xFFFFFFFFu && ((lanes & (lanes - 1u)) | many)) {
        // equal ranks: the smallest (key, tie) of the lane's, then of the warp's
        const bool ex = exact(mw);  // the keys are equal too
        uint64_t kk = psk::kNoKey;
        bt = 0xFFFFFFFFu;
#pragma unroll
        for (int k = 0; k < IPT; ++k)
          if (rank[k] == mw) {
            const uint2 w = key_words(k);
            const uint64_t x = ex ? 0ull : pair_key<GEN>(m, mw, w, h[k]);
            if (x < kk || (x == kk && tie[k] < bt)) {
              kk = x;
              bk = w;
              bt = tie[k];
              bh = h[k];
            }
          }
        const int win = ex ? __ffs(__ballot_sync(0xffffffffu, bt == __reduce_min_sync(0xffffffffu, bt))) - 1
                           : warp_argmin(has ? mw : 0xFFFFFFFFu, kk, bt);
        __syncwarp();
        if (lane == win) {
          s_th[s & 1u][warp] = make_uint2(bt, bh);
          s_key[s & 1u][warp] = bk;
        }
      }
      __syncwarp();
    }
    if (!stopped) {
#pragma unroll
      for (int k = 0; k < IPT; ++k) {  // the pending state: each owner's instances
        const uint32_t i = i0 + (uint32_t)k;
        if (i < I) {
          pending.b[i] = committed.b[i];
          pending.qr[i] = (int32_t)(kq[k] & 0x3FFFFu);
          pending.q[i] = q32[k];
          pending.S[i] = S32[k];
          pending.M[i] = committed.M[i];
          pending.Bmax[i] = committed.Bmax[i];
        }
      }
    }
  } else {
    // ---- compute warps, 64-bit sums: some q or S may leave [0, 2^30) ---------------------------------
    // The same steps with every order's key, and the shared-memory truth for sums that need 64 bits.
    int32_t room[IPT], q32[IPT], S32[IPT], Bp[IPT];
    float dec0[IPT], fe[IPT], tq[IPT];
    uint64_t kd[IPT];
    bool wide = false;  // some q or S of this thread's instances is outside [0, 2^30): 64-bit sums from shared memory
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
      const uint32_t i = i0 + (uint32_t)k;
      room[k] = -1;
      q32[k] = S32[k] = 0;
      Bp[k] = 1;
      dec0[k] = fe[k] = tq[k] = 0.0f;
      kd[k] = 0ull;
      if (i < I) {
        const psk::InstTerms it = psk::inst_terms(m, a.b[i], a.qr[i], a.q[i], a.Bmax[i]);
        room[k] = it.okB ? psk::kv_room(a.S[i], a.M[i]) : -1;
        dec0[k] = it.dec0;
        fe[k] = it.f;
        tq[k] = it.tq;
        Bp[k] = it.Bp;
        kd[k] = psk::dcq_key0(a.b[i], a.qr[i]);
        q32[k] = (int32_t)a.q[i];
        S32[k] = (int32_t)a.S[i];
        wide |= !narrow_qs(a.q[i], a.S[i]);
      }
    }
    uint32_t Lprev = 0;  // length of request s - 1
    for (uint32_t s = 0;; ++s) {
      bar_step();
      if (s_stop <= s) {
        stopped = true;
        break;
      }
      const uint32_t slot = (s < R ? s : R - 1) % kFeedRing;
      uint32_t own = 0xFFFFFFFFu;  // this thread's index of the last pick, if it owns it
      uint32_t lj = 0;             // what its hit on this row rises to
      if (s > 0) {
        const int src = decision(s - 1, rank_of(s - 1));
        const uint2 th = s_th[(s - 1) & 1u][src < 0 ? 0 : src];
        const uint32_t j = th.x & psk::kTieInstMask;
        lj = s_row[slot].lcp[0];
        if (LIN && src >= 0 && j / (32u * IPT) == warp) lj = extend(s_row[slot], j, s_hitr[slot * Ip + j]);
        if (src >= 0 && j / IPT == t) {
          own = j - i0;
          const int32_t b = a.b[j], qr = a.qr[j] + 1;
          const int64_t q = a.q[j] + (int64_t)Lprev - 16 * (int64_t)th.y;
          const int64_t S = a.S[j] + (int64_t)Lprev;
          a.qr[j] = qr;
          a.q[j] = q;
          a.S[j] = S;
          const psk::InstTerms it = psk::inst_terms(m, b, qr, q, a.Bmax[j]);
          const int32_t rm = it.okB ? psk::kv_room(S, a.M[j]) : -1;
          wide |= !narrow_qs(q, S);
#pragma unroll
          for (int k = 0; k < IPT; ++k)
            if ((uint32_t)k == own) {
              room[k] = rm;
              q32[k] = (int32_t)q;
              S32[k] = (int32_t)S;
              Bp[k] = it.Bp;
              dec0[k] = it.dec0;
              fe[k] = it.f;
              tq[k] = it.tq;
              kd[k] += 1ull;  // qr + 1
            }
        }
      }
      if (s == R) break;
      const psk::RowPre& row = s_row[slot];
      const StepRow rc = step_row(row);
      Lprev = rc.L;
      uint32_t h[IPT], tb[IPT];
      if (loads) {
        lds_words<IPT>(s_hitr + slot * Ip + i0, h);
        lds_words<IPT>(s_tpfr + slot * Ip + i0, tb);
      } else {
#pragma unroll
        for (int k = 0; k < IPT; ++k) h[k] = tb[k] = 0u;
      }
      if (own != 0xFFFFFFFFu) {  // the last pick also took request s - 1: its common prefix with this row
        const uint32_t tl = __float_as_uint(psk::t_pf32(m, rc.L, lj));
#pragma unroll
        for (int k = 0; k < IPT; ++k)
          if ((uint32_t)k == own && lj > h[k]) {
            h[k] = lj;
            tb[k] = tl;
          }
      }
      // every pair: W, the capacity guard, the latencies, and the key it has in C
      float W[IPT];
      uint64_t key[IPT];
      uint32_t tie[IPT];
      float wbest = INFINITY;
#pragma unroll
      for (int k = 0; k < IPT; ++k) {
        const uint32_t i = i0 + (uint32_t)k < I ? i0 + (uint32_t)k : 0u;
        const float tpf = __uint_as_float(tb[k]);
        const int32_t n = (int32_t)rc.L - (int32_t)(h[k] << 4);
        W[k] = (int32_t)rc.L <= room[k] ? __fsub_rn(tpf, rc.t_cached) : INFINITY;
        wbest = fminf(wbest, W[k]);
        psk::RowConst rr;
        rr.L = rc.L;
        rr.tpot_target = rc.tpot_target;
        float tpot, ttft;
        uint64_t qn;
        if (!wide) {
          psk::pair_lat32(m, rr, tpf, n, dec0[k], fe[k], tq[k], Bp[k], q32[k], S32[k], &tpot, &ttft);
          qn = (uint64_t)(uint32_t)(q32[k] + n);
        } else {
          psk::InstTerms it;
          it.dec0 = dec0[k];
          it.f = fe[k];
          it.tq = tq[k];
          it.Bp = Bp[k];
          it.okB = 1;
          psk::PairW x;
          x.W = W[k];
          x.tpf = tpf;
          x.n = n;
          x.inA = true;
          psk::pair_lat(m, rr, x, it, a.q[i], a.S[i], &tpot, &ttft);
          qn = (uint64_t)a.q[i] + (uint64_t)(int64_t)n;
        }
        const bool adm = (tpot < rc.tpot_lim) & (ttft <= rc.ttft_max);
        tie[k] = i0 + (uint32_t)k;
        if (adm) {
          key[k] = psk::packed_key(0u, psk::value_in_t(m, psk::key0_from_dcq(m, kd[k]), h[k], tpot, rc.tpot_target));
          if (m.sel == psk::kSelHCQ) tie[k] |= (uint32_t)(kd[k] & 0x3FFFFull) << 12;
        } else {
          key[k] = psk::packed_key(1u, psk::value_fallback(m, qn, (uint32_t)Bp[k], kd[k], h[k]));
        }
      }
      uint32_t wmin_o = __reduce_min_sync(0xffffffffu, psk::f2ord(wbest));
      if (ncw > 1u) {
        if (lane == 0) s_w[warp] = wmin_o;
        bar_compute();
        wmin_o = __reduce_min_sync(0xffffffffu, s_w[lane & (kComputeWarps - 1)]);
      }
      const float wmin = psk::ord2f(wmin_o);
      // the recompute filter (a pair outside A has W = +infinity, and W - W_min = +infinity or NaN), then
      // this thread's smallest (key, tie)
      uint64_t bk[IPT];
      uint32_t bt[IPT], bh[IPT];
#pragma unroll
      for (int k = 0; k < IPT; ++k) {
        const bool in = __fsub_rn(W[k], wmin) <= rc.c_max;
        bk[k] = in ? key[k] : psk::kNoKey;
        bt[k] = tie[k];
        bh[k] = h[k];
      }
#pragma unroll
      for (int d = 1; d < IPT; d <<= 1)
#pragma unroll
        for (int k = 0; k < IPT; k += 2 * d) {
          const bool less = bk[k + d] < bk[k] || (bk[k + d] == bk[k] && bt[k + d] < bt[k]);
          bk[k] = less ? bk[k + d] : bk[k];
          bt[k] = less ? bt[k + d] : bt[k];
          bh[k] = less ? bh[k + d] : bh[k];
        }
      const uint32_t rank = key_rank(bk[0]);
      const int win = warp_argmin(rank, bk[0], bt[0]);
      if (lane == (win < 0 ? 0 : win)) {
        s_rank[s & 1u][warp] = rank;
        s_th[s & 1u][warp] = make_uint2(bt[0], bh[0]);
        s_key[s & 1u][warp] = make_uint2((uint32_t)bk[0], (uint32_t)(bk[0] >> 32));
      }
      __syncwarp();
    }
    if (!stopped) {
#pragma unroll
      for (int k = 0; k < IPT; ++k) {
        const uint32_t i = i0 + (uint32_t)k;
        if (i < I) {
          pending.b[i] = a.b[i];
          pending.qr[i] = a.qr[i];
          pending.q[i] = a.q[i];
          pending.S[i] = a.S[i];
          pending.M[i] = a.M[i];
          pending.Bmax[i] = a.Bmax[i];
        }
      }
    }
  }
  if (t == 0 && sync.stats) {
    atomicAdd(sync.stats + psk::kGsDecisions, (unsigned long long)(stopped ? 0u : R));
    atomicAdd(sync.stats + psk::kGsDecideTotal, (unsigned long long)(clock64() - cyc0));
  }
}

// GEN: not Algorithm 1's order (Table 4 / Table 3 variants); EQ9: Eq. 9's interference term; LIN: caches that are
// not prefix-closed (built for every order).
template <int IPT, bool GEN, bool EQ9, bool LIN>
__global__ void __launch_bounds__(kPipeThreads, 1)
greedy_pipe_kernel(const psk::RowPre* __restrict__ rows, const uint64_t* __restrict__ hash, uint32_t R, uint32_t I,
                   const uint32_t* __restrict__ hit0, const float* __restrict__ tpf0, psk::StateSoA committed,
                   psk::StateSoA pending, psk::DevModel m, psk::DeltaSlot* delta, uint64_t nslots, int32_t* assign,
                   uint8_t* __restrict__ path, uint32_t* __restrict__ hit_chosen, uint32_t* err, psk::GreedySync sync,
                   uint32_t ninsert, MainTables mt, uint64_t tokens) {
  extern __shared__ __align__(16) unsigned long long smem_raw[];
  if (blockIdx.x == 0) {
    decide_rows<IPT, GEN, EQ9, LIN>(rows, R, I, committed, pending, m, assign, path, hit_chosen, err, sync, smem_raw, hash, mt,
                                    tokens);
  } else if (blockIdx.x <= ninsert) {
    insert_blocks<LIN>(rows, hash, R, delta, nslots, err, sync, blockIdx.x - 1, ninsert);
  } else {
    probe_rows<IPT, LIN>(rows, hash, R, I, hit0, tpf0, m, delta, nslots, err, sync, smem_raw, blockIdx.x - 1 - ninsert,
                         gridDim.x - 1 - ninsert, mt);
  }
}

size_t greedy_pipe_smem(uint32_t I, uint32_t Ip) {
  // deciding block: instance state, the hit and T_pf rows of kFeedRing rows; probe blocks: three u32
  // arrays per instance
  const size_t decide = (size_t)Ip * (kInstSmemBytes + 2 * kFeedRing * sizeof(uint32_t));
  const size_t probe = (size_t)I * 3 * sizeof(uint32_t);
  return decide > probe ? decide : probe;
}

template <int IPT>
cudaError_t greedy_pipe_launch(const psk::RowPre* rows, const psk::WindowDev& w, uint32_t I, const uint32_t* hit0,
                               const float* tpf0, psk::StateSoA committed, psk::StateSoA pending, const psk::DevModel& m,
                               psk::DeltaSlot* delta, uint64_t nslots, int32_t* assign, uint8_t* path,
                               uint32_t* hit_chosen, uint32_t* err, const psk::GreedySync& sync, bool linear,
                               MainTables mt, uint64_t tokens, int num_sms, cudaStream_t s) {
  const bool gen = m.sel != psk::kSelDCQ || m.fb_dcq, eq9 = m.interference_mode != 0;
  decltype(&greedy_pipe_kernel<IPT, true, true, true>) kern;
  if (linear) kern = eq9 ? greedy_pipe_kernel<IPT, true, true, true> : greedy_pipe_kernel<IPT, true, false, true>;
  else if (gen) kern = eq9 ? greedy_pipe_kernel<IPT, true, true, false> : greedy_pipe_kernel<IPT, true, false, false>;
  else kern = eq9 ? greedy_pipe_kernel<IPT, false, true, false> : greedy_pipe_kernel<IPT, false, false, false>;
  const size_t smem = greedy_pipe_smem(I, sync.ring_stride);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const uint64_t* hash = w.hash;
  uint32_t R = w.R;
  psk::StateSoA c = committed, p = pending;
  psk::DevModel mm = m;
  psk::GreedySync sy = sync;
  uint32_t ninsert = 0;
  void* args[] = {(void*)&rows, (void*)&hash, (void*)&R, (void*)&I, (void*)&hit0, (void*)&tpf0, (void*)&c, (void*)&p,
                  (void*)&mm, (void*)&delta, (void*)&nslots, (void*)&assign, (void*)&path, (void*)&hit_chosen,
                  (void*)&err, (void*)&sy, (void*)&ninsert, (void*)&mt, (void*)&tokens};
  // All blocks must be resident at once, and one fits on an SM.  A stream may be limited to fewer SMs than the
  // device reports: a launch that is too large for it is refused before it starts, and half as many tried.
  for (uint32_t resident = (uint32_t)num_sms;; resident /= 2u) {
    const psgrid::PipeGrid g = psgrid::pipe_grid(R, psk::kLag, resident);
    ninsert = g.insert;
    e = cudaLaunchCooperativeKernel((const void*)kern, dim3(g.blocks()), dim3(kPipeThreads), args, smem, s);
    if (e != cudaErrorCooperativeLaunchTooLarge || g.blocks() <= psgrid::kMinBlocks) return e;
    cudaGetLastError();
  }
}

}  // namespace

namespace pskl {

cudaError_t launch_greedy(const psk::RowPre* rows, const psk::WindowDev& w, uint32_t I, const uint32_t* hit0,
                                 const float* tpf0, psk::StateSoA committed, psk::StateSoA pending, const psk::DevModel& m,
                                 psk::DeltaSlot* delta, uint64_t delta_nslots, int32_t* assign, uint8_t* path,
                                 uint32_t* hit_chosen, uint32_t* err, const psk::GreedySync& sync, int search,
                                 const uint64_t* slots, const uint64_t* ovf, const psk::TableDesc* tdesc,
                                 uint64_t win_blocks, int num_sms, cudaStream_t s) {
  const MainTables mt{slots, ovf, tdesc};
  const cudaError_t e = cudaMemsetAsync(sync.stats, 0, sync.clear_bytes, s);
  if (e != cudaSuccess || w.R == 0) return e;
  // IPT instances per compute thread of the deciding block (and at most that many per probe thread): as
  // few as its warps allow.  More per thread means fewer warps to combine but a longer step: greedy pass
  // with 1 / 2 / 4 a thread 0.32 / 0.33 / 0.44 ms at 256 x 512, with 2 / 4 / 8 14.6 / 17.0 / 25.2 at 1024 x 16384.
  const uint32_t ipt = (I + 32u * kComputeWarps - 1) / (32u * kComputeWarps);
#define PS_GREEDY_P(IPT)                                                                                      \
  return greedy_pipe_launch<IPT>(rows, w, I, hit0, tpf0, committed, pending, m, delta, delta_nslots, assign, path, \
                                 hit_chosen, err, sync, search == 0, mt, 16u * (win_blocks + w.R), num_sms, s)
  if (ipt <= 1) PS_GREEDY_P(1);
  if (ipt <= 2) PS_GREEDY_P(2);
  if (ipt <= 4) PS_GREEDY_P(4);
#undef PS_GREEDY_P
  return cudaErrorInvalidValue;
}

// The delta table only holds one window's blocks: clear it whole after each window.
cudaError_t launch_delta_clear(psk::DeltaSlot* delta, uint64_t nslots, cudaStream_t s) {
  return cudaMemsetAsync(delta, 0, nslots * sizeof(psk::DeltaSlot), s);
}

}  // namespace pskl
