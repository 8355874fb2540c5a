// Table maintenance and between-window kernels: bulk insertion of cached chains, commit of a
// scheduled window, engine progress of a streaming window, leaf-first LRU eviction, the
// prefix-closure check and the device-side window layout check.
#include "ps_internal.cuh"

namespace {

// Bulk insert: one thread block per instance, the table's only writer.  Block 0 of chain c continues
// parent[c], block k continues block k - 1.  The result is that of inserting the chains' blocks one
// after another: the block collects its instance's chains in order (kInsThreads list entries per step)
// and takes their blocks kInsThreads at a time, all positions of a tile at once:
//   find    every position looks its key up in the table (and a chain's first block its parent);
//   dedupe  the keys not found meet in a hash set in shared memory, the lowest position of each wins;
//   place   the winners claim slots by compare-and-swap: the emptier candidate bucket first (as just
//           read), and the overflow run of the table's layout when both are full;
//   link    with LRU metadata, each new block records its parent's slot and the parent gains a child;
//           a parent counts if it was cached before the block in the order above.
// Bound by the dependent round trips of a tile (about 3 to L2 or memory), not by bandwidth: one warp
// inserting block after block took 2.1 us a block.  Bringing up a context with 96 instances x 20000
// blocks took 46.6 ms that way, 0.89 ms now.
constexpr uint32_t kInsThreads = 512;
constexpr uint32_t kInsQueue = 2 * kInsThreads;  // chains collected before their blocks are inserted
constexpr uint32_t kInsSet = 2 * kInsThreads;    // hash set of a tile's new keys (a power of two)

// Claims a slot for a key that is not in the table, while other threads insert other keys.  v, the
// key's two candidate buckets as last read, only chooses where to try first.  ~0: the table is full.
__device__ uint64_t place_key(uint64_t* slots, uint64_t* ovf, const psk::TableDesc& d, uint64_t key,
                              const psk::Lookup& L) {
  const uint32_t b1 = L.b1, b2 = psk::fastrange32(psk::remix(key), d.nbkt);
  uint32_t e1 = 0u, e2 = 0u;  // empty slots of each bucket, one bit each
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    e1 |= (L.v[k].x == psk::kEmpty ? 1u : 0u) << (2 * k) | (L.v[k].y == psk::kEmpty ? 2u : 0u) << (2 * k);
    e2 |= (L.v[4 + k].x == psk::kEmpty ? 1u : 0u) << (2 * k) | (L.v[4 + k].y == psk::kEmpty ? 2u : 0u) << (2 * k);
  }
  const bool first1 = __popc(e1) >= __popc(e2);  // the emptier bucket, b1 on ties
#pragma unroll 1
  for (int c = 0; c < 2; ++c) {
    const bool one = (c == 0) == first1;
    unsigned long long* base =
        reinterpret_cast<unsigned long long*>(slots + d.base + (uint64_t)(one ? b1 : b2) * psk::kBucketSlots);
    for (uint32_t e = one ? e1 : e2; e; e &= e - 1u) {  // slots never empty again: only the empty ones matter
      const int k = __ffs(e) - 1;
      if (atomicCAS(base + k, (unsigned long long)psk::kEmpty, (unsigned long long)key) == psk::kEmpty)
        return (uint64_t)(base + k - reinterpret_cast<unsigned long long*>(slots));
    }
  }
  uint32_t b = b1;
  for (uint32_t step = 0; step < d.nbkt; ++step) {
    atomicOr(reinterpret_cast<unsigned long long*>(ovf + d.ovf + (b >> 6)), 1ull << (b & 63));
    b = (b + 1 == d.nbkt) ? 0u : b + 1;
    unsigned long long* base = reinterpret_cast<unsigned long long*>(slots + d.base + (uint64_t)b * psk::kBucketSlots);
    for (int k = 0; k < psk::kBucketSlots; ++k)
      if (__ldcg(base + k) == psk::kEmpty &&
          atomicCAS(base + k, (unsigned long long)psk::kEmpty, (unsigned long long)key) == psk::kEmpty)
        return (uint64_t)(base + k - reinterpret_cast<unsigned long long*>(slots));
  }
  return ~0ull;
}

struct InsSmem {
  uint64_t start[kInsQueue];     // a collected chain's first block in the hash array
  uint64_t pre[kInsQueue];       // its first position among the collected blocks
  uint64_t chain[kInsQueue];     // its index
  unsigned long long key[kInsSet];
  uint32_t pos[kInsSet];         // lowest position (thread) of the key in the tile
  uint64_t slot[kInsThreads];    // slot of each position's block (~0: none)
  uint32_t wsum[kInsThreads / 32];
  unsigned long long wlen[kInsThreads / 32];
  uint64_t carry;                // slot of the block before the tile's first position
  unsigned long long added;
};

// Index of key in the tile's set, or kInsSet if absent (the set holds at most half its size).
__device__ __forceinline__ uint32_t set_find(const InsSmem& s, uint64_t key) {
  for (uint32_t h = (uint32_t)(key >> 20) & (kInsSet - 1), p = 0; p < kInsSet; ++p, h = (h + 1) & (kInsSet - 1)) {
    if (s.key[h] == key) return h;
    if (s.key[h] == psk::kEmpty) return kInsSet;
  }
  return kInsSet;
}

__global__ void __launch_bounds__(kInsThreads)
insert_chains_kernel(uint64_t* slots, uint64_t* ovf, const psk::TableDesc* __restrict__ tdesc, uint32_t I,
                     unsigned long long* count, uint64_t nchains, const uint32_t* __restrict__ inst,
                     const uint64_t* __restrict__ off, const uint64_t* __restrict__ hash,
                     const uint64_t* __restrict__ parent, psk::LruMeta meta, uint32_t last_use, uint32_t* err) {
  extern __shared__ __align__(16) unsigned char ins_raw[];
  InsSmem& s = *reinterpret_cast<InsSmem*>(ins_raw);
  const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  for (uint32_t i = blockIdx.x; i < I; i += gridDim.x) {
    const psk::TableDesc d = tdesc[i];
    uint32_t nq = 0;      // collected chains and blocks (block-uniform)
    uint64_t nblk = 0;
    bool full = false, reserved = false;
    if (t == 0) {
      s.added = 0ull;
      s.carry = ~0ull;
    }
    __syncthreads();
    uint32_t next = t < nchains ? __ldg(inst + t) : 0xFFFFFFFFu;
    for (uint64_t c0 = 0; c0 < nchains; c0 += kInsThreads) {
      const uint64_t c = c0 + t;
      const bool mine = c < nchains && next == i;
      const uint64_t cn = c + kInsThreads;
      next = cn < nchains ? __ldg(inst + cn) : 0xFFFFFFFFu;
      const bool last = c0 + kInsThreads >= nchains;
      if (__syncthreads_or(mine ? 1 : 0)) {
        // append this step's chains in order: exclusive sums of (chains, blocks) over the threads
        const uint64_t a = mine ? __ldg(off + c) : 0ull;
        const unsigned long long len = mine ? __ldg(off + c + 1) - a : 0ull;
        const unsigned bal = __ballot_sync(0xffffffffu, mine);
        unsigned long long x = len;
#pragma unroll
        for (int dd = 1; dd < 32; dd <<= 1) {
          const unsigned long long y = __shfl_up_sync(0xffffffffu, x, dd);
          if (lane >= (uint32_t)dd) x += y;
        }
        if (lane == 31u) {
          s.wsum[warp] = __popc(bal);
          s.wlen[warp] = x;
        }
        __syncthreads();
        uint32_t bn = 0, tn = 0;
        unsigned long long bl = 0, tl = 0;
#pragma unroll
        for (uint32_t v = 0; v < kInsThreads / 32; ++v) {
          if (v == warp) {
            bn = tn;
            bl = tl;
          }
          tn += s.wsum[v];
          tl += s.wlen[v];
        }
        if (mine) {
          const uint32_t at = nq + bn + __popc(bal & ((1u << lane) - 1u));
          s.start[at] = a;
          s.pre[at] = nblk + bl + x - len;
          s.chain[at] = c;
        }
        nq += tn;
        nblk += tl;
        __syncthreads();
      }
      if (!last && nq <= kInsQueue - kInsThreads && nblk < 8ull * kInsThreads) continue;
      for (uint64_t p0 = 0; p0 < nblk; p0 += kInsThreads) {
        const uint64_t p = p0 + t;
        for (uint32_t x = t; x < kInsSet; x += kInsThreads) {
          s.key[x] = psk::kEmpty;
          s.pos[x] = 0xFFFFFFFFu;
        }
        uint32_t e = 0;  // the position's chain: the last one that begins at or before it
        uint64_t key = psk::kEmpty;
        bool first = false;
        if (p < nblk) {
          uint32_t hi = nq;
          while (hi - e > 1u) {
            const uint32_t mid = (e + hi) >> 1;
            if (s.pre[mid] <= p) e = mid;
            else hi = mid;
          }
          first = s.pre[e] == p;
          key = __ldg(hash + s.start[e] + (p - s.pre[e]));
          reserved |= key == psk::kEmpty || key == psk::kTomb;
        }
        const bool live = key != psk::kEmpty && key != psk::kTomb;
        // find: the table as the earlier tiles left it
        psk::Lookup L;
        uint64_t slot = ~0ull;
        const uint64_t pkey = first && meta.last_use ? __ldg(parent + s.chain[e]) : psk::kEmpty;
        uint64_t pslot = ~0ull;
        if (live) {
          psk::lookup_issue<false>(slots, ovf, d, key, L);
          if (psk::lookup_finish<false>(slots, ovf, d, key, L)) slot = psk::main_find(slots, ovf, d, key);
        }
        if (pkey != psk::kEmpty) pslot = psk::main_find(slots, ovf, d, pkey);
        __syncthreads();
        // dedupe: positions of one new key agree on the lowest
        uint32_t h = kInsSet;
        if (live && slot == ~0ull) {
          h = (uint32_t)(key >> 20) & (kInsSet - 1);
          for (;;) {  // at most kInsThreads keys: a free entry comes within kInsSet steps
            const unsigned long long old = atomicCAS(&s.key[h], (unsigned long long)psk::kEmpty, (unsigned long long)key);
            if (old == psk::kEmpty || old == key) break;
            h = (h + 1) & (kInsSet - 1);
          }
          atomicMin(&s.pos[h], t);
        }
        __syncthreads();
        const bool winner = h < kInsSet && s.pos[h] == t;
        bool stored = false;
        if (winner) {
          slot = place_key(slots, ovf, d, key, L);
          if (slot == ~0ull) {
            full = true;
          } else {
            stored = true;
            if (meta.last_use) {
              meta.last_use[slot] = last_use;
              meta.children[slot] = 0u;
            }
          }
        } else if (slot != ~0ull && meta.last_use && meta.last_use[slot] < last_use) {
          meta.last_use[slot] = last_use;
        }
        const unsigned ns = __popc(__ballot_sync(0xffffffffu, stored));
        if (lane == 0 && ns) atomicAdd(&s.added, (unsigned long long)ns);
        if (meta.last_use) {
          s.slot[t] = slot;
          __syncthreads();
          if (h < kInsSet && !winner) slot = s.slot[s.pos[h]];  // the winner's slot
          const uint64_t carry = s.carry;
          __syncthreads();
          s.slot[t] = slot;
          __syncthreads();
          if (stored) {
            if (!first) {
              pslot = t > 0 ? s.slot[t - 1] : carry;
            } else if (pslot == ~0ull && pkey != psk::kEmpty && pkey != psk::kTomb) {
              const uint32_t q = set_find(s, pkey);  // inserted by this tile, at an earlier position
              if (q < kInsSet && s.pos[q] < t) pslot = s.slot[s.pos[q]];
            }
            meta.parent[slot] = pslot == ~0ull ? psk::kNoParent : pslot;
            if (pslot != ~0ull) atomicAdd(meta.children + pslot, 1u);
          }
          if (t == kInsThreads - 1u) s.carry = slot;
        }
        __syncthreads();  // the next tile reuses the set and reads what this one stored
      }
      nq = 0;
      nblk = 0;
      __syncthreads();
    }
    if (t == 0) count[i] += s.added;
    if (full) atomicOr(err, psk::kErrTableFull);
    if (reserved) atomicOr(err, psk::kErrReservedHash);
    __syncthreads();
  }
}

// Instance ids must be valid before the per-instance scan (a chain with a bad id is never seen).
__global__ void check_instances_kernel(uint32_t I, uint64_t nchains, const uint32_t* __restrict__ inst,
                                       uint32_t* err) {
  for (uint64_t c = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; c < nchains; c += (uint64_t)gridDim.x * blockDim.x)
    if (inst[c] >= I) atomicOr(err, psk::kErrBadInstance);
}

// Commit of a scheduled window, in four passes over every admitted request's blocks (within a window
// each (block, instance) pair is inserted at most once: a request inserts chain[h, nb) on its pick
// with h the exact first miss there, so none of those blocks is cached on that instance yet, neither
// by the committed caches nor by an earlier request):
//   stamp   the cached prefix chain[0, h) gets last_use (every stamp writes the same value, so
//           their order does not matter);
//   insert  the uncached blocks chain[h, nb) are cached, stamped, with 0 children and their parent
//           link pending;
//   link    each new block records its parent's slot and the parent gains a child;
//   queue   with request tracking, each instance appends its admitted requests to its FIFO queue
//           in arrival order (one warp per instance).
// The first three run over one flat index space of (request, block) items, so a long chain is
// spread over the whole grid: a prefix pass gives each admitted request its first item, and an item
// finds its request by binary search.

// Exclusive prefix sums over the window's requests of the items of the stamp pass (h) and of the
// insert and link passes (nb - h); rejected requests have none.  One block; pre_s and pre_i hold
// R + 1 entries each.
__global__ void __launch_bounds__(1024)
commit_prefix_kernel(psk::WindowDev w, const int32_t* __restrict__ assign, const uint32_t* __restrict__ hit_chosen,
                     unsigned long long* pre_s, unsigned long long* pre_i) {
  __shared__ unsigned long long s_ws[32], s_wi[32];
  __shared__ unsigned long long s_carry_s, s_carry_i;
  const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  if (t == 0) {
    s_carry_s = 0ull;
    s_carry_i = 0ull;
  }
  __syncthreads();
  for (uint32_t r0 = 0; r0 < w.R; r0 += blockDim.x) {
    const uint32_t r = r0 + t;
    unsigned long long cs = 0ull, ci = 0ull;
    if (r < w.R && assign[r] >= 0) {
      const uint64_t h = hit_chosen[r];
      const uint64_t nb = w.off[r + 1] - w.off[r];
      cs = h;
      ci = nb > h ? nb - h : 0ull;
    }
    unsigned long long xs = cs, xi = ci;  // inclusive warp scans
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned long long ys = __shfl_up_sync(0xffffffffu, xs, d), yi = __shfl_up_sync(0xffffffffu, xi, d);
      if ((int)lane >= d) {
        xs += ys;
        xi += yi;
      }
    }
    if (lane == 31u) {
      s_ws[warp] = xs;
      s_wi[warp] = xi;
    }
    __syncthreads();
    if (warp == 0) {
      const uint32_t nw = blockDim.x >> 5;
      unsigned long long vs = lane < nw ? s_ws[lane] : 0ull, vi = lane < nw ? s_wi[lane] : 0ull;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long ys = __shfl_up_sync(0xffffffffu, vs, d), yi = __shfl_up_sync(0xffffffffu, vi, d);
        if ((int)lane >= d) {
          vs += ys;
          vi += yi;
        }
      }
      // exclusive warp offsets from the inclusive ones
      const unsigned long long es = __shfl_up_sync(0xffffffffu, vs, 1), ei = __shfl_up_sync(0xffffffffu, vi, 1);
      if (lane < nw) {
        s_ws[lane] = lane == 0 ? 0ull : es;
        s_wi[lane] = lane == 0 ? 0ull : ei;
      }
    }
    __syncthreads();
    if (r < w.R) {
      pre_s[r] = s_carry_s + s_ws[warp] + xs - cs;
      pre_i[r] = s_carry_i + s_wi[warp] + xi - ci;
    }
    __syncthreads();
    if (t == blockDim.x - 1u) {  // the chunk's total carries into the next chunk
      s_carry_s += s_ws[warp] + xs;
      s_carry_i += s_wi[warp] + xi;
    }
    __syncthreads();
  }
  if (t == 0) {
    pre_s[w.R] = s_carry_s;
    pre_i[w.R] = s_carry_i;
  }
}

// The request of flat item x: the last r with pre[r] <= x (pre ascending, pre[0] = 0, x < pre[R]).
__device__ __forceinline__ uint32_t item_request(const unsigned long long* __restrict__ pre, uint32_t R,
                                                 unsigned long long x) {
  uint32_t lo = 0, hi = R;  // pre[lo] <= x < pre[hi]
  while (hi - lo > 1u) {
    const uint32_t mid = (lo + hi) >> 1;
    if (__ldg(pre + mid) <= x) lo = mid;
    else hi = mid;
  }
  return lo;
}

__global__ void commit_stamp_kernel(const uint64_t* slots, const uint64_t* ovf, const psk::TableDesc* __restrict__ tdesc,
                                    psk::WindowDev w, const int32_t* __restrict__ assign,
                                    const unsigned long long* __restrict__ pre_s, psk::LruMeta meta, uint32_t last_use) {
  const unsigned long long total = pre_s[w.R];
  for (unsigned long long x = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; x < total;
       x += (unsigned long long)gridDim.x * blockDim.x) {
    const uint32_t r = item_request(pre_s, w.R, x);
    const uint64_t k = x - pre_s[r];
    const uint64_t s = psk::main_find(slots, ovf, tdesc[assign[r]], w.hash[w.off[r] + k]);
    if (s != ~0ull && meta.last_use[s] < last_use) meta.last_use[s] = last_use;
  }
}

__global__ void commit_insert_kernel(uint64_t* slots, uint64_t* ovf, const psk::TableDesc* __restrict__ tdesc,
                                     unsigned long long* count, psk::WindowDev w, const int32_t* __restrict__ assign,
                                     const uint32_t* __restrict__ hit_chosen, const unsigned long long* __restrict__ pre_i,
                                     psk::LruMeta meta, uint32_t last_use, uint32_t* err) {
  const unsigned long long total = pre_i[w.R];
  for (unsigned long long x = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; x < total;
       x += (unsigned long long)gridDim.x * blockDim.x) {
    const uint32_t r = item_request(pre_i, w.R, x);
    const int32_t j = assign[r];
    const uint64_t k = hit_chosen[r] + (x - pre_i[r]);
    const uint64_t key = w.hash[w.off[r] + k];
    if (key == psk::kEmpty || key == psk::kTomb) continue;
    bool ins = false;
    const uint64_t slot = psk::thread_insert(slots, ovf, tdesc[j], key, &ins);
    if (slot == ~0ull) {
      atomicOr(err, psk::kErrTableFull);
      continue;
    }
    if (ins) {
      atomicAdd(count + j, 1ull);
      if (meta.last_use) {
        meta.last_use[slot] = last_use;
        meta.children[slot] = 0;
        meta.parent[slot] = psk::kLinkPending;
      }
    } else if (meta.last_use && meta.last_use[slot] < last_use) {
      meta.last_use[slot] = last_use;
    }
  }
}

__global__ void commit_link_kernel(const uint64_t* slots, const uint64_t* ovf, const psk::TableDesc* __restrict__ tdesc,
                                   psk::WindowDev w, const int32_t* __restrict__ assign,
                                   const uint32_t* __restrict__ hit_chosen, const unsigned long long* __restrict__ pre_i,
                                   psk::LruMeta meta) {
  const unsigned long long total = pre_i[w.R];
  for (unsigned long long x = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; x < total;
       x += (unsigned long long)gridDim.x * blockDim.x) {
    const uint32_t r = item_request(pre_i, w.R, x);
    const psk::TableDesc d = tdesc[assign[r]];
    const uint64_t o = w.off[r];
    const uint64_t k = hit_chosen[r] + (x - pre_i[r]);
    const uint64_t key = w.hash[o + k];
    const uint64_t pkey = k > 0 ? w.hash[o + k - 1] : psk::kEmpty;
    const uint64_t s = psk::main_find(slots, ovf, d, key);
    if (s == ~0ull || meta.parent[s] != psk::kLinkPending) continue;  // not inserted by this commit
    const uint64_t ps = k > 0 ? psk::main_find(slots, ovf, d, pkey) : ~0ull;
    meta.parent[s] = ps == ~0ull ? psk::kNoParent : ps;
    if (ps != ~0ull) atomicAdd(meta.children + ps, 1u);
  }
}

__global__ void commit_queue_kernel(uint32_t I, psk::WindowDev w, const int32_t* __restrict__ assign,
                                    const uint32_t* __restrict__ hit_chosen, psk::ReqStore rq,
                                    const uint32_t* __restrict__ out_tokens, uint32_t* err) {
  const int lane = threadIdx.x & 31;
  const uint32_t warps_total = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < I; i += warps_total) {
    bool overflow = false;
    for (uint32_t r0 = 0; r0 < w.R; r0 += 32) {
      const uint32_t r = r0 + lane;
      unsigned mine = __ballot_sync(0xffffffffu, r < w.R && assign[r] == (int32_t)i);
      while (mine) {  // in arrival order
        const uint32_t rr = r0 + (uint32_t)(__ffs(mine) - 1);
        mine &= mine - 1;
        if (lane == 0) {
          const uint32_t len = rq.q_len[i];
          if (len >= rq.M) {
            overflow = true;
          } else {
            const uint64_t at = (uint64_t)i * rq.M + (rq.q_head[i] + len) % rq.M;
            rq.q_L[at] = w.L[rr];
            rq.q_out[at] = out_tokens ? out_tokens[rr] : 0u;
            rq.q_rem[at] = (uint64_t)((int64_t)w.L[rr] - 16 * (int64_t)hit_chosen[rr]);
            rq.q_len[i] = len + 1;
          }
        }
        __syncwarp();
      }
    }
    if (lane == 0 && overflow) atomicOr(err, psk::kErrRequestsFull);
  }
}

// Engine progress of one streaming window, one warp per instance (the serving engine's rules):
// every decoding request emits k = max(1, floor(window_ms / ((b0 + b1 b) + b2 S))) tokens (fp32,
// state at the window start), finished requests leave (b -= 1, S -= L + out), then the FIFO queue
// drains prefill_tokens tokens and requests whose prefill completes start decoding.
__global__ void advance_kernel(psk::StateSoA st, uint32_t I, psk::ReqStore rq, psk::DevModel m, float window_ms,
                               uint64_t prefill_tokens, uint32_t* err) {
  const int lane = threadIdx.x & 31;
  const uint32_t warps_total = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < I; i += warps_total) {
    int32_t b = st.b[i], qr = st.qr[i];
    int64_t q = st.q[i], S = st.S[i];
    float t_iter = __fadd_rn(m.b0, __fmul_rn(m.b1, __int2float_rn(b)));
    t_iter = __fadd_rn(t_iter, __fmul_rn(m.b2, __ll2float_rn(S)));
    const float per = __fdiv_rn(window_ms, t_iter);
    int64_t kk = (int64_t)per;  // per > 0: truncation is floor
    if (kk < 1) kk = 1;
    const uint32_t k = kk > 0xFFFFFFFFll ? 0xFFFFFFFFu : (uint32_t)kk;
    // decode progress with in-warp compaction of the survivors
    const uint32_t n = rq.d_len[i];
    const uint64_t base = (uint64_t)i * rq.M;
    uint32_t kept = 0;
    int64_t dS = 0;
    int32_t done = 0;
    for (uint32_t x0 = 0; x0 < n; x0 += 32) {
      const uint32_t x = x0 + lane;
      uint32_t L = 0, out = 0, rem = 0;
      bool live = false;
      if (x < n) {
        L = rq.d_L[base + x];
        out = rq.d_out[base + x];
        rem = rq.d_rem[base + x];
        const uint32_t e = rem < k ? rem : k;
        rem -= e;
        dS += e;
        live = rem > 0;
        if (!live) {
          done += 1;
          dS -= (int64_t)L + (int64_t)out;
        }
      }
      const unsigned lv = __ballot_sync(0xffffffffu, live);
      __syncwarp();
      if (live) {
        const uint32_t at = kept + __popc(lv & ((1u << lane) - 1u));
        rq.d_L[base + at] = L;
        rq.d_out[base + at] = out;
        rq.d_rem[base + at] = rem;
      }
      kept += __popc(lv);
      __syncwarp();
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
      dS += __shfl_xor_sync(0xffffffffu, dS, s);
      done += __shfl_xor_sync(0xffffffffu, done, s);
    }
    S += dS;
    b -= done;
    if (lane == 0) {
      uint32_t len = rq.q_len[i], head = rq.q_head[i];
      uint64_t budget = prefill_tokens;
      uint32_t dl = kept;
      bool overflow = false;
      while (budget > 0 && len > 0) {
        const uint64_t at = base + head;
        const uint64_t rem = rq.q_rem[at];
        const uint64_t take = rem < budget ? rem : budget;
        rq.q_rem[at] = rem - take;
        q -= (int64_t)take;
        budget -= take;
        if (rem == take) {
          if (dl < rq.M) {
            rq.d_L[base + dl] = rq.q_L[at];
            rq.d_out[base + dl] = rq.q_out[at];
            rq.d_rem[base + dl] = rq.q_out[at];
            ++dl;
          } else {
            overflow = true;
          }
          head = (head + 1) % rq.M;
          --len;
          qr -= 1;
          b += 1;
        }
      }
      rq.q_len[i] = len;
      rq.q_head[i] = head;
      rq.d_len[i] = dl;
      st.b[i] = b;
      st.qr[i] = qr;
      st.q[i] = q;
      st.S[i] = S;
      if (overflow) atomicOr(err, psk::kErrRequestsFull);
    }
  }
}

// A leaf candidate with its parent's slot (kLeafNoParent for none), so that evicting it needs no
// dependent load before the parent's metadata can be read.  Five 32-bit words (the hash split).
struct Leaf {
  uint32_t last_use;
  uint32_t slot;
  uint32_t hash_lo, hash_hi;
  uint32_t parent;
};
static_assert(sizeof(Leaf) == 20, "a leaf is five 32-bit words");
constexpr uint32_t kLeafNoParent = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t parent32(uint64_t p) {
  return (p == psk::kNoParent || p == psk::kLinkPending) ? kLeafNoParent : (uint32_t)p;
}

// Leaf-first LRU eviction of the instances over capacity.
//
// Evicting the smallest leaf by (last_use, hash) again and again removes blocks in increasing order of
// their subtree maximum of (last_use, hash), deeper first where two share it.  Where stamps never
// increase down a chain (a commit stamps a request's whole chain, a bulk insert every block it touches)
// a block's subtree maximum has its own last_use.  So with T the last_use value at which the blocks
// counted from the oldest reach the excess E, the evicted blocks are exactly: every block older than T,
// and of the blocks stamped T the k missing ones with the smallest subtree maximum of the hash over
// blocks stamped T.  These kernels find and evict them, every step parallel:
//   list      the instances over capacity (or, where every excess is small, flags them for the kernels after
//             these);
//   hist      per instance a histogram of last_use over its slots (and its number of leaves), in one
//             pass for stamps below 2048 and one more per further 11 bits; choose picks T and k;
//   gather    the slots stamped below T and those stamped T (up to kClassMax each; at most kClassMax
//             evictions a round);
//   detail    every gathered block's parent, children count and the parent's stamp, and the hashes of
//             the class T, side by side (the metadata is scattered, a DRAM access each: this wants
//             every warp of the chip), with the sums of the check that the stamps do not increase
//             downwards among these blocks and that none of them has a newer child;
//   index, jump  each class block's index in place of its (known) stamp, then its parent's index;
//   order     one thread block per instance finds the subtree maxima of the class T by doubling over the
//             parent links in shared memory (a block pushes its maximum to its ancestor 2^r links up in
//             round r); selects the k smallest; evicts.
// At most kEvictBatch instances a round.
// An instance that fails the check, or has more blocks stamped T than shared memory holds, is evicted
// one block at a time by the kernels after these.  Bound by the two scans (last_use twice and the
// children counts once: 12 bytes a slot; an empty slot's stamp is kNoUse, so the keys are not read)
// and the order kernel's chain of dependent steps.  1024 instances x 200K blocks, about 240 over
// capacity by up to 7.9K blocks: hist 0.12 ms, gather 0.11, detail 0.09, index and jump 0.07, order 0.17
// (0.43 ms where the order kernel read the metadata itself, a block an SM); the streaming window of 500
// requests takes 1.59 ms, and took 11.8 ms with one thread ordering each instance's evictions (1.2 us each).
// That is a cache filled by commits, or loaded with many stamps.  One loaded with a single stamp gains nothing
// until its first blocks are gone: 200K blocks of one stamp an instance are more than kClassMax, so the scan
// and the choice find that out (0.1 ms) and the kernels below do the work; advancing such a stream of
// 1000-request windows takes 15.0 ms a window over the first 13 (15.0 with those kernels alone), 7.8 over 1000
// (7.7); one of 4 instances over by 300 blocks, 0.65 ms (0.58).
constexpr uint32_t kClassMax = 16384;   // blocks of one last_use value ordered in shared memory
constexpr uint32_t kHistBits = 11;
constexpr uint32_t kHistBins = 1u << kHistBits;
constexpr uint32_t kOrderThreads = 1024;
constexpr uint32_t kOrderPer = kClassMax / kOrderThreads;  // class blocks per thread
constexpr uint32_t kScanThreads = 512;
constexpr uint64_t kScanChunk = 65536;  // slots a block scans before it merges its histogram
constexpr uint32_t kNoJump = 0xFFFFu;
static_assert(kClassMax < kNoJump, "16-bit block indices");
// Bits of the "another round" word: instances left for these kernels, for the one-at-a-time kernels; and
// whether this call's list had any for these.
constexpr uint32_t kMoreFast = 1u, kMoreSlow = 2u, kMoreListed = 4u;
// Excess up to which every instance of a call goes block by block (and half the number of instances over
// capacity more): that is 0.7 us a block on one thread, all instances side by side, against the launches and
// steps of the class kernels.  A call's time, one by one / by classes: 2 of 8 instances over by 5 blocks
// 55 / 101 us, by 64 about 97 / 101, by 200 193 / 91; 256 of 1024 over by 20 129 / 262, by 192 about 250 / 265.
constexpr uint32_t kSmallExcess = 64u;

// Per over-capacity instance: the last_use range still open, what was counted below it, and the choice.
struct EvictPlan {
  uint32_t lo, hi;       // T lies in [lo, hi]
  uint32_t below;        // blocks stamped below lo
  uint32_t todo;         // evictions of this round
  uint32_t k;            // of them, blocks stamped T (T = lo once chosen)
  uint32_t n_old, n_cls; // gathered blocks
  uint32_t leaves;
  uint32_t children, inside, bad;  // the check's sums: cached children of the gathered blocks, gathered
                                   // blocks with a gathered parent; some child is newer than its parent
  __device__ bool fits() const { return k != 0u && n_old <= kClassMax && n_cls <= kClassMax; }
  __device__ bool in_order() const { return bad == 0u && children == inside; }
};

// The gathered blocks of the q-th listed instance: [0, kClassMax) stamped below T, [kClassMax, 2
// kClassMax) stamped T (the class).
constexpr uint32_t kEvictBatch = 256;
struct EvictBlocks {
  uint32_t* slot;   // [kEvictBatch][2 kClassMax]
  uint32_t* par;    // the parent's slot
  uint8_t* rel;     // the parent's stamp against T: kRel*
  uint64_t* key;    // [kEvictBatch][kClassMax] the class's hashes
  uint16_t* jump;   // [kEvictBatch][kClassMax] index of the parent in the class (kNoJump: none)
};
enum : uint8_t { kRelNone = 0, kRelOlder = 1, kRelClass = 2, kRelNewer = 3 };


// Also starts the round word and, in a call's first round, the flags and the leaf counts.
__global__ void __launch_bounds__(1024)
evict_list_kernel(uint32_t I, const unsigned long long* __restrict__ count, const uint64_t* __restrict__ cap,
                  uint32_t* slow, uint32_t* nleaf, uint32_t max_use, EvictPlan* plan, uint32_t* list, uint32_t* nlist,
                  uint32_t* more, bool first, bool class_runs) {
  __shared__ uint32_t s_n, s_over;
  __shared__ unsigned long long s_excess;
  if (threadIdx.x == 0) {
    s_n = 0u;
    s_over = 0u;
    s_excess = 0ull;
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < I; i += blockDim.x) {
    if (first) slow[i] = nleaf[i] = 0u;
    if (count[i] > cap[i] && !slow[i]) {
      atomicAdd(&s_over, 1u);
      atomicMax(&s_excess, count[i] - cap[i]);
    }
  }
  __syncthreads();
  const bool small = s_excess <= kSmallExcess + s_over / 2u;
  for (uint32_t i = threadIdx.x; i < I; i += blockDim.x) {
    const unsigned long long c = count[i];
    if (c <= cap[i] || slow[i]) continue;
    if (small) {
      slow[i] = 1u;
      continue;
    }
    const uint32_t q = atomicAdd(&s_n, 1u);
    if (q >= kEvictBatch) continue;
    const unsigned long long E = c - cap[i];
    EvictPlan p{};
    p.hi = max_use;
    p.todo = E < kClassMax ? (uint32_t)E : kClassMax;
    plan[i] = p;
    list[q] = i;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    *nlist = s_n < kEvictBatch ? s_n : kEvictBatch;
    const bool left = class_runs ? s_n > kEvictBatch : s_n > 0u;
    *more = (s_n ? kMoreListed : 0u) | (left ? kMoreFast : 0u) | (small && s_over && class_runs ? kMoreSlow : 0u);
  }
}

// Bin width of an open range as a shift.
__device__ __forceinline__ uint32_t hist_shift(uint32_t lo, uint32_t hi) {
  const uint32_t span = hi - lo;
  return span < kHistBins ? 0u : 32u - (uint32_t)__clz(span) - kHistBits;
}

__global__ void __launch_bounds__(kScanThreads)
evict_hist_kernel(const psk::TableDesc* __restrict__ tdesc, psk::LruMeta meta,
                  EvictPlan* plan, const uint32_t* __restrict__ list, const uint32_t* __restrict__ nlist,
                  uint64_t chunks, uint32_t* __restrict__ hist, bool first) {
  __shared__ uint32_t s_bin[kHistBins];
  __shared__ uint32_t s_leaves;
  const uint64_t items = (uint64_t)*nlist * chunks;
  for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const uint32_t q = (uint32_t)(item / chunks), i = list[q];
    const psk::TableDesc d = tdesc[i];
    const uint64_t n = (uint64_t)d.nbkt * psk::kBucketSlots, x0 = (item % chunks) * kScanChunk;
    if (x0 >= n) continue;  // block-uniform
    const uint64_t x1 = x0 + kScanChunk < n ? x0 + kScanChunk : n;
    const uint32_t lo = plan[i].lo, hi = plan[i].hi, sh = hist_shift(lo, hi);
    for (uint32_t b = threadIdx.x; b < kHistBins; b += kScanThreads) s_bin[b] = 0u;
    if (threadIdx.x == 0) s_leaves = 0u;
    __syncthreads();
    uint32_t leaves = 0;
    // four slots a thread (tables are whole 8-slot buckets); an empty slot's stamp says so
    for (uint64_t x = x0 + 4u * threadIdx.x; x < x1; x += 4u * kScanThreads) {
      const uint4 lu = __ldcs(reinterpret_cast<const uint4*>(meta.last_use + d.base + x));
      uint4 ch = make_uint4(1u, 1u, 1u, 1u);
      if (first) ch = __ldcs(reinterpret_cast<const uint4*>(meta.children + d.base + x));
      const uint32_t l[4] = {lu.x, lu.y, lu.z, lu.w}, cc[4] = {ch.x, ch.y, ch.z, ch.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (l[u] == psk::kNoUse) continue;
        if (l[u] >= lo && l[u] <= hi) atomicAdd(&s_bin[(l[u] - lo) >> sh], 1u);
        leaves += cc[u] == 0u;
      }
    }
    if (first) {
      leaves = __reduce_add_sync(0xffffffffu, leaves);
      if ((threadIdx.x & 31u) == 0u && leaves) atomicAdd(&s_leaves, leaves);
    }
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < kHistBins; b += kScanThreads)
      if (s_bin[b]) atomicAdd(&hist[(uint64_t)q * kHistBins + b], s_bin[b]);
    if (first && threadIdx.x == 0) atomicAdd(&plan[i].leaves, s_leaves);
    __syncthreads();
  }
}

// Narrows the open range to the bin in which the count reaches the round's evictions; with one value
// a bin that value is T.  Clears the histogram for the next pass.
__global__ void __launch_bounds__(256)
evict_choose_kernel(EvictPlan* plan, const uint32_t* __restrict__ list, const uint32_t* __restrict__ nlist,
                    uint32_t* __restrict__ hist) {
  constexpr uint32_t kPer = kHistBins / 256;
  __shared__ uint32_t s_sum[256];
  const uint32_t t = threadIdx.x;
  for (uint32_t x = blockIdx.x; x < *nlist; x += gridDim.x) {
    const uint32_t i = list[x];
    const EvictPlan p = plan[i];
    const uint32_t sh = hist_shift(p.lo, p.hi);
    uint32_t v[kPer], sum = 0;
#pragma unroll
    for (uint32_t u = 0; u < kPer; ++u) {
      uint32_t* b = &hist[(uint64_t)x * kHistBins + t * kPer + u];
      v[u] = *b;
      *b = 0u;
      sum += v[u];
    }
    s_sum[t] = sum;
    __syncthreads();
    for (uint32_t dd = 1; dd < 256; dd <<= 1) {
      const uint32_t y = t >= dd ? s_sum[t - dd] : 0u;
      __syncthreads();
      s_sum[t] += y;
      __syncthreads();
    }
    uint32_t acc = p.below + s_sum[t] - sum;  // blocks stamped below this thread's bins
#pragma unroll
    for (uint32_t u = 0; u < kPer; ++u) {
      if (acc < p.todo && acc + v[u] >= p.todo) {  // one thread, one bin
        const uint32_t lo = p.lo + ((t * kPer + u) << sh);
        const uint32_t w = (1u << sh) - 1u;
        plan[i].lo = lo;
        plan[i].hi = p.hi - lo < w ? p.hi : lo + w;
        plan[i].below = acc;
        plan[i].k = sh == 0u && v[u] > kClassMax ? 0u : p.todo - acc;  // too many for the order kernel: not gathered
      }
      acc += v[u];
    }
    __syncthreads();
  }
}

// Gathers the slots stamped below T (first half of the instance's candidate buffer) and T (second half).
__global__ void __launch_bounds__(kScanThreads)
evict_gather_kernel(const psk::TableDesc* __restrict__ tdesc, psk::LruMeta meta,
                    EvictPlan* plan, const uint32_t* __restrict__ list, const uint32_t* __restrict__ nlist,
                    uint64_t chunks, EvictBlocks eb) {
  const uint64_t items = (uint64_t)*nlist * chunks;
  const uint32_t lane = threadIdx.x & 31u;
  for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const uint32_t i = list[item / chunks];
    if (plan[i].k == 0u) continue;  // block-uniform
    const psk::TableDesc d = tdesc[i];
    const uint64_t n = (uint64_t)d.nbkt * psk::kBucketSlots, x0 = (item % chunks) * kScanChunk;
    const uint64_t x1 = x0 + kScanChunk < n ? x0 + kScanChunk : n;
    const uint32_t T = plan[i].lo;
    uint32_t* out = eb.slot + (item / chunks) * 2u * kClassMax;
    for (uint64_t xb = x0; xb < x1; xb += 4u * kScanThreads) {  // (tables are whole 8-slot buckets)
      const uint64_t x = xb + 4u * threadIdx.x;
      uint4 lu = make_uint4(psk::kNoUse, psk::kNoUse, psk::kNoUse, psk::kNoUse);
      if (x < x1) lu = __ldcs(reinterpret_cast<const uint4*>(meta.last_use + d.base + x));
      const uint32_t l[4] = {lu.x, lu.y, lu.z, lu.w};
      uint32_t oldm = 0u, clsm = 0u;
#pragma unroll
      for (int u = 0; u < 4; ++u) {  // (T is never the mark of an empty slot)
        oldm |= (l[u] < T ? 1u : 0u) << u;
        clsm |= (l[u] == T ? 1u : 0u) << u;
      }
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const uint32_t mask = half ? clsm : oldm;
        const uint32_t mine = __popc(mask);
        if (!__any_sync(0xffffffffu, mine != 0u)) continue;
        uint32_t sum = mine;
#pragma unroll
        for (int dd = 1; dd < 32; dd <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, sum, dd);
          if (lane >= (uint32_t)dd) sum += y;
        }
        uint32_t at = 0;
        if (lane == 31u) at = atomicAdd(half ? &plan[i].n_cls : &plan[i].n_old, sum);
        at = __shfl_sync(0xffffffffu, at, 31) + sum - mine;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if ((mask >> u) & 1u) {
            if (at < kClassMax) out[half * kClassMax + at] = (uint32_t)(d.base + x) + u;
            ++at;
          }
      }
    }
  }
}

constexpr uint32_t kDetailThreads = 512;

__global__ void __launch_bounds__(kDetailThreads)
evict_detail_kernel(const uint64_t* __restrict__ slots, psk::LruMeta meta, EvictPlan* plan,
                    const uint32_t* __restrict__ list, const uint32_t* __restrict__ nlist, EvictBlocks eb) {
  constexpr uint32_t kChunks = 2u * kClassMax / kDetailThreads;
  const uint32_t items = *nlist * kChunks;
  for (uint32_t item = blockIdx.x; item < items; item += gridDim.x) {
    const uint32_t q = item / kChunks, x0 = (item % kChunks) * kDetailThreads;
    const uint32_t i = list[q];
    const EvictPlan p = plan[i];
    const bool cls = x0 >= kClassMax;
    const uint32_t n = cls ? p.n_cls : p.n_old, x = (cls ? x0 - kClassMax : x0) + threadIdx.x;
    if (!p.fits() || (cls ? x0 - kClassMax : x0) >= n) continue;  // block-uniform
    uint32_t ch = 0u, in = 0u;
    bool bad = false;
    if (x < n) {
      const uint64_t at = (uint64_t)q * 2u * kClassMax + x0 + threadIdx.x;
      const uint32_t sl = eb.slot[at];
      ch = meta.children[sl];
      const uint32_t ps = parent32(meta.parent[sl]);
      const uint32_t lu = cls ? p.lo : meta.last_use[sl];
      if (cls) eb.key[(uint64_t)q * kClassMax + x] = slots[sl];
      uint8_t rel = kRelNone;
      if (ps != kLeafNoParent) {
        const uint32_t lp = meta.last_use[ps];
        rel = lp < p.lo ? kRelOlder : (lp == p.lo ? kRelClass : kRelNewer);
        in = lp <= p.lo;
        bad = lp < lu;
      }
      eb.par[at] = ps;
      eb.rel[at] = rel;
    }
    ch = __reduce_add_sync(0xffffffffu, ch);
    in = __reduce_add_sync(0xffffffffu, in);
    const bool anybad = __any_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31u) == 0u) {
      if (ch) atomicAdd(&plan[i].children, ch);
      if (in) atomicAdd(&plan[i].inside, in);
      if (anybad) atomicOr(&plan[i].bad, 1u);
    }
  }
}

// JUMP false: a class block's index stands in for its (known) stamp; true: its parent's index is read.
template <bool JUMP>
__global__ void __launch_bounds__(kDetailThreads)
evict_index_kernel(psk::LruMeta meta, const EvictPlan* __restrict__ plan, const uint32_t* __restrict__ list,
                   const uint32_t* __restrict__ nlist, uint32_t max_leaves, EvictBlocks eb) {
  constexpr uint32_t kChunks = kClassMax / kDetailThreads;
  const uint32_t items = *nlist * kChunks;
  for (uint32_t item = blockIdx.x; item < items; item += gridDim.x) {
    const uint32_t q = item / kChunks, x = (item % kChunks) * kDetailThreads + threadIdx.x;
    const EvictPlan& p = plan[list[q]];
    if (!p.fits() || !p.in_order() || p.leaves > max_leaves || p.k >= p.n_cls || x >= p.n_cls) continue;
    const uint64_t at = (uint64_t)q * 2u * kClassMax + kClassMax + x;
    if (!JUMP) meta.last_use[eb.slot[at]] = x;
    else
      eb.jump[(uint64_t)q * kClassMax + x] =
          (uint16_t)(eb.rel[at] == kRelClass ? meta.last_use[eb.par[at]] : kNoJump);
  }
}

struct OrderSmem {
  unsigned long long M[kClassMax];  // subtree maximum of the hash over the class
  uint16_t jump[kClassMax];         // ancestor 2^r links up (kNoJump: past the class)
  uint16_t dep[kClassMax];          // links to the topmost ancestor in the class, plus one
  uint32_t hist[256];
  unsigned long long sel;           // radix selection: the chosen bytes so far
  uint32_t rank;                    // and the rank among the values that share them
  uint32_t dep_max;
};

__global__ void __launch_bounds__(kOrderThreads)
evict_order_kernel(uint64_t* slots, unsigned long long* count, const uint64_t* __restrict__ cap, psk::LruMeta meta,
                   const EvictPlan* __restrict__ plan, const uint32_t* __restrict__ list,
                   const uint32_t* __restrict__ nlist, EvictBlocks eb, uint32_t* slow, uint32_t* more,
                   uint32_t max_leaves, uint32_t* err) {
  extern __shared__ __align__(16) unsigned char order_raw[];
  OrderSmem& s = *reinterpret_cast<OrderSmem*>(order_raw);
  const uint32_t t = threadIdx.x;
  for (uint32_t item = blockIdx.x; item < *nlist; item += gridDim.x) {
    const uint32_t i = list[item];
    const EvictPlan p = plan[i];
    const uint32_t T = p.lo, n = p.n_cls, n_old = p.n_old;
    if (p.leaves > max_leaves) {  // (the limit of the one-at-a-time kernels, kept for every instance)
      if (t == 0) {
        atomicOr(err, psk::kErrLeavesFull);
        slow[i] = 2u;  // not evicted in this call
      }
      continue;
    }
    if (!p.fits() || !p.in_order()) {
      if (t == 0) {
        slow[i] = 1u;
        atomicOr(more, kMoreSlow);
      }
      continue;
    }
    const uint32_t* old_slots = eb.slot + (uint64_t)item * 2u * kClassMax;
    const uint32_t* cls_slots = old_slots + kClassMax;
    const uint32_t* old_par = eb.par + (uint64_t)item * 2u * kClassMax;
    const uint32_t* cls_par = old_par + kClassMax;
    const uint8_t* old_rel = eb.rel + (uint64_t)item * 2u * kClassMax;
    const uint8_t* cls_rel = old_rel + kClassMax;
    const bool whole = p.k >= n;
    uint32_t gone = 0u;  // bit u: this thread's class block t + u kOrderThreads is evicted
    if (whole) {
      gone = (1u << kOrderPer) - 1u;
    } else {
#pragma unroll
      for (uint32_t u = 0; u < kOrderPer; ++u) {
        const uint32_t x = t + u * kOrderThreads;
        if (x < n) {
          s.M[x] = eb.key[(uint64_t)item * kClassMax + x];
          s.jump[x] = eb.jump[(uint64_t)item * kClassMax + x];
          s.dep[x] = 1;
        }
      }
      __syncthreads();
      for (;;) {  // at most 14 rounds: a path holds at most kClassMax blocks
        uint32_t nj[kOrderPer];
        uint32_t nd[kOrderPer];
        bool any = false;
#pragma unroll
        for (uint32_t u = 0; u < kOrderPer; ++u) {
          const uint32_t x = t + u * kOrderThreads;
          nj[u] = kNoJump;
          nd[u] = 0u;
          if (x < n && s.jump[x] != kNoJump) {
            const uint32_t j = s.jump[x];
            any = true;
            const unsigned long long v = s.M[x];
            if (s.M[j] < v) atomicMax(&s.M[j], v);
            nj[u] = s.jump[j];
            nd[u] = s.dep[j];
          }
        }
        if (!__syncthreads_or(any ? 1 : 0)) break;
#pragma unroll
        for (uint32_t u = 0; u < kOrderPer; ++u) {
          const uint32_t x = t + u * kOrderThreads;
          if (x < n && s.jump[x] != kNoJump) {
            s.jump[x] = (uint16_t)nj[u];
            s.dep[x] = (uint16_t)(s.dep[x] + nd[u]);
          }
        }
        __syncthreads();
      }
      // the k-th smallest maximum, byte by byte from the top
      if (t == 0) {
        s.sel = 0ull;
        s.rank = p.k - 1u;
        s.dep_max = 0u;
      }
      for (int sh = 56; sh >= 0; sh -= 8) {
        if (t < 256) s.hist[t] = 0u;
        __syncthreads();
        const unsigned long long sel = s.sel;
        const unsigned long long high = sh == 56 ? 0ull : ~0ull << (sh + 8);
#pragma unroll
        for (uint32_t u = 0; u < kOrderPer; ++u) {
          const uint32_t x = t + u * kOrderThreads;
          // maxima crowd into few values of the upper bytes: a warp of one value adds once
          const unsigned long long v = x < n ? s.M[x] : 0ull;
          const bool in = x < n && (v & high) == sel;
          const uint32_t digit = in ? (uint32_t)(v >> sh) & 255u : 256u;
          const unsigned im = __ballot_sync(0xffffffffu, in);
          if (im == 0u) continue;
          const uint32_t d0 = __shfl_sync(0xffffffffu, digit, __ffs(im) - 1);
          if (__all_sync(0xffffffffu, !in || digit == d0)) {
            if ((t & 31u) == (uint32_t)__ffs(im) - 1u) atomicAdd(&s.hist[d0], (uint32_t)__popc(im));
          } else if (in) {
            atomicAdd(&s.hist[digit], 1u);
          }
        }
        __syncthreads();
        if (t < 32) {  // the bin that holds the rank
          uint32_t v[8], sum = 0;
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            v[u] = s.hist[t * 8 + u];
            sum += v[u];
          }
          uint32_t x = sum;
#pragma unroll
          for (int dd = 1; dd < 32; dd <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, dd);
            if ((int)t >= dd) x += y;
          }
          const uint32_t rank = s.rank;
          uint32_t acc = x - sum;
          __syncwarp();
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            if (acc <= rank && rank < acc + v[u]) {  // one lane, one bin
              s.sel = sel | ((unsigned long long)(t * 8 + u) << sh);
              s.rank = rank - acc;
            }
            acc += v[u];
          }
        }
        __syncthreads();
      }
      // blocks that share the k-th maximum lie on one path, the deepest (whose hash it is) first
      const unsigned long long cut = s.sel;
      const uint32_t rank = s.rank;
#pragma unroll
      for (uint32_t u = 0; u < kOrderPer; ++u) {
        const uint32_t x = t + u * kOrderThreads;
        if (x < n && s.M[x] == cut) atomicMax(&s.dep_max, (uint32_t)s.dep[x]);
      }
      __syncthreads();
      const uint32_t dm = s.dep_max;
#pragma unroll
      for (uint32_t u = 0; u < kOrderPer; ++u) {
        const uint32_t x = t + u * kOrderThreads;
        if (x < n && (s.M[x] < cut || (s.M[x] == cut && s.dep[x] + rank >= dm))) gone |= 1u << u;
      }
    }
    // evict: the slots first, then the counts of the parents that stay (an evicted slot keeps its links:
    // whoever fills it sets its parent and children)
#pragma unroll
    for (uint32_t u = 0; u < kOrderPer; ++u) {
      const uint32_t x = t + u * kOrderThreads;
      if (x >= n) continue;
      const bool g = (gone >> u) & 1u;
      if (g) slots[cls_slots[x]] = psk::kEmpty;
      if (g || !whole) meta.last_use[cls_slots[x]] = g ? psk::kNoUse : T;
    }
    for (uint32_t x = t; x < n_old; x += kOrderThreads) {
      slots[old_slots[x]] = psk::kEmpty;
      meta.last_use[old_slots[x]] = psk::kNoUse;
    }
    __syncthreads();
    auto drop = [&](uint32_t ps, uint8_t rel) {
      if (rel == kRelNewer || (rel == kRelClass && !whole && __ldcg(slots + ps) != psk::kEmpty))
        atomicSub(meta.children + ps, 1u);
    };
#pragma unroll
    for (uint32_t u = 0; u < kOrderPer; ++u) {
      const uint32_t x = t + u * kOrderThreads;
      if (x < n && ((gone >> u) & 1u)) drop(cls_par[x], cls_rel[x]);
    }
    for (uint32_t x = t; x < n_old; x += kOrderThreads) drop(old_par[x], old_rel[x]);
    if (t == 0) {
      const unsigned long long c = count[i] - p.todo;
      count[i] = c;
      if (c > cap[i]) atomicOr(more, kMoreFast);
    }
    __syncthreads();
  }
}

// One block at a time (instances flagged slow), in rounds of two kernels:
//   collect  all SMs scan the over-capacity instances' slots (coalesced) and append each leaf (a
//            cached block with no cached child) to its instance's leaf buffer;
//   evict    one thread block per over-capacity instance sorts its leaves by (last_use, hash), then
//            thread 0 evicts in order, taking the smaller of the next sorted leaf and the smallest
//            parent that became a leaf (a small heap); the parent is reached through its stored slot.
// Every evicted block only ever makes its parent a leaf, and a leaf outside the first E sorted ones
// can never be among E evictions, so a round of at most kHeapMax evictions reproduces the
// one-at-a-time rule exactly; the host repeats rounds while an instance is still over capacity.
//
// A loader warp reads each parent's metadata from global memory ahead of the ordered loop: for the
// sorted leaves, up to kRing leaves past the loop's position; for a parent that became a leaf, as
// soon as it is pushed.  The loop never waits for it: a record not filled yet is read by the loop
// itself, with the same result.  Children counts are not written during the loop, so every read
// sees the round's starting count; the loop keeps the decremented counts in a shared hash table,
// written back at the end of the round.  A block's metadata changes in a round only when it is
// evicted, which happens after every record that names it as a parent has been read.  Most
// evictions climb a chain (a parent goes right after its last child, when its key is below the next
// candidate's); such a step reads its record itself, since the parent's parent is known only from
// the parent's metadata.
constexpr int kLeafMax = 4096;
constexpr int kHeapMax = 1536;
constexpr int kEvictThreads = 256;
constexpr int kRing = 32;          // sorted leaves whose parent records the loader keeps ready
constexpr int kDeltaSlots = 2048;  // children counts a round changes (at most kHeapMax parents)
constexpr uint64_t kEvictWaitNs = 1000000000ull;  // bound on the loader's idle wait
static_assert(kHeapMax < kDeltaSlots, "the count table never fills");
constexpr int kCollectThreads = 256;
constexpr uint32_t kCollectSlotsPerThread = 8;

__device__ __forceinline__ Leaf make_leaf(uint32_t last_use, uint32_t slot, uint64_t hash, uint64_t parent) {
  return Leaf{last_use, slot, (uint32_t)hash, (uint32_t)(hash >> 32), parent32(parent)};
}

__device__ __forceinline__ bool leaf_less(const Leaf& a, const Leaf& b) {
  if (a.last_use != b.last_use) return a.last_use < b.last_use;
  return a.hash_hi != b.hash_hi ? a.hash_hi < b.hash_hi : a.hash_lo < b.hash_lo;
}

__device__ __forceinline__ void heap_push(Leaf* h, int& n, const Leaf& x) {
  int c = n++;
  h[c] = x;
  while (c > 0) {
    const int p = (c - 1) >> 1;
    if (!leaf_less(h[c], h[p])) break;
    const Leaf t = h[c];
    h[c] = h[p];
    h[p] = t;
    c = p;
  }
}

__device__ __forceinline__ Leaf heap_pop(Leaf* h, int& n) {
  const Leaf top = h[0];
  h[0] = h[--n];
  int c = 0;
  for (;;) {
    const int l = 2 * c + 1, r = l + 1;
    int m = c;
    if (l < n && leaf_less(h[l], h[m])) m = l;
    if (r < n && leaf_less(h[r], h[m])) m = r;
    if (m == c) break;
    const Leaf t = h[c];
    h[c] = h[m];
    h[m] = t;
    c = m;
  }
  return top;
}

// A parent's metadata as the loader reads it: children count at the start of the round, last_use,
// hash and its own parent's slot.  A pool record also holds the slot it describes (a parent that
// became a leaf names its record by index, in the heap entry's parent word).
struct ParentRec {
  uint32_t pc, plu, ph_lo, ph_hi, ppp;
};
struct PoolRec {
  uint32_t pp;
  ParentRec r;
};
static_assert(sizeof(ParentRec) == 20 && sizeof(PoolRec) == 24, "records are 32-bit words");

// Shared memory of an eviction block.  The sort uses all kLeafMax leaves; a round then reads only
// the first kHeapMax sorted ones, and the rest of that space holds the records and the count table.
constexpr size_t kOffPool = (size_t)kHeapMax * sizeof(Leaf);
constexpr size_t kOffRing = kOffPool + (size_t)kHeapMax * sizeof(PoolRec);
constexpr size_t kOffDKey = kOffRing + (size_t)kRing * sizeof(ParentRec);
constexpr size_t kOffDVal = kOffDKey + (size_t)kDeltaSlots * sizeof(uint32_t);
constexpr size_t kOffHeapRaw = kOffDVal + (size_t)kDeltaSlots * sizeof(uint32_t);
constexpr size_t kOffHeap =
    kOffHeapRaw > (size_t)kLeafMax * sizeof(Leaf) ? kOffHeapRaw : (size_t)kLeafMax * sizeof(Leaf);
constexpr size_t kEvictSmem = kOffHeap + (size_t)kHeapMax * sizeof(Leaf);
// two eviction blocks per SM: 2 x (kEvictSmem + the static flags + 1 KB reserved) <= 228 KB
static_assert(2 * (kEvictSmem + 64 + 1024) <= 228 * 1024, "two eviction blocks fit on an SM");
__device__ __forceinline__ ParentRec load_parent(const uint64_t* slots, const psk::LruMeta& meta, uint32_t ps) {
  ParentRec r{0u, 0u, 0u, 0u, kLeafNoParent};
  if (ps != kLeafNoParent) {
    const uint32_t pc = meta.children[ps], plu = meta.last_use[ps];
    const uint64_t ph = slots[ps], pp = meta.parent[ps];
    r = ParentRec{pc, plu, (uint32_t)ph, (uint32_t)(ph >> 32), parent32(pp)};
  }
  return r;
}
// The decremented children count of ps (first touch: from the round's starting count pc).
__device__ __forceinline__ uint32_t count_dec(uint32_t* dkey, uint32_t* dval, uint32_t ps, uint32_t pc) {
  uint32_t h = (ps * 0x9E3779B1u) >> 21;  // 11 bits: kDeltaSlots entries
  for (int probe = 0; probe < kDeltaSlots; ++probe) {
    const uint32_t k = dkey[h];
    if (k == ps) return --dval[h];
    if (k == kLeafNoParent) {
      dkey[h] = ps;
      dval[h] = pc - 1u;
      return pc - 1u;
    }
    h = (h + 1u) & (uint32_t)(kDeltaSlots - 1);
  }
  return 1u;  // not reached: a round changes fewer counts than the table holds
}
static_assert(kDeltaSlots == 1 << 11, "count_dec hashes to 11 bits");

struct EvictFlags {
  uint32_t ptr;        // sorted leaves the loop has taken (their records may be overwritten)
  uint32_t ring_done;  // sorted leaves whose parent records are in the ring
  uint32_t req;        // pool records the loop has asked for
  uint32_t pool_done;  // pool records filled
  uint32_t exit;       // the loop has ended
};

// The loader warp: fills ring records for sorted leaves [ring_done, min(m, ptr + kRing)) and pool
// records [pool_done, req), one record of each kind per lane per pass, loads issued before any
// record is written.  Every control value is the warp's minimum of what its lanes observed, so the
// warp stays converged and each lane's acquire covers what it reads.
__device__ void evict_loader(const uint64_t* slots, const psk::LruMeta& meta, const Leaf* leaves, ParentRec* ring,
                             PoolRec* pool, uint32_t m, EvictFlags* f, uint32_t* err) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t ring_done = 0, pool_done = 0;
  const long long c0 = clock64();
  const long long lim = (long long)(kEvictWaitNs * 3ull);
  for (uint32_t it = 1;; ++it) {
    uint32_t ex = psk::ld_relaxed_cta_shared_u32(&f->exit);
    uint32_t ptr = psk::ld_relaxed_cta_shared_u32(&f->ptr);
    uint32_t req = psk::ld_relaxed_cta_shared_u32(&f->req);
    psk::fence_acq_rel_cta();
    ex = __reduce_min_sync(0xffffffffu, ex);
    ptr = __reduce_min_sync(0xffffffffu, ptr);
    req = __reduce_min_sync(0xffffffffu, req);
    if (ex) return;
    const uint32_t rhi = ptr + (uint32_t)kRing < m ? ptr + (uint32_t)kRing : m;
    const uint32_t phi = req < pool_done + 32u ? req : pool_done + 32u;
    if (ring_done >= rhi && pool_done >= phi) {
      if ((it & 31u) == 0u && __any_sync(0xffffffffu, clock64() - c0 > lim)) {
        if (lane == 0) atomicOr(err, psk::kErrTimeout);
        return;
      }
      continue;
    }
    const uint32_t j = ring_done + lane, k = pool_done + lane;
    const bool rj = j < rhi, pk = k < phi;
    const ParentRec a = load_parent(slots, meta, rj ? leaves[j].parent : kLeafNoParent);
    const uint32_t pp = pk ? pool[k].pp : kLeafNoParent;
    const ParentRec b = load_parent(slots, meta, pp);
    if (rj) ring[j % (uint32_t)kRing] = a;
    if (pk) pool[k].r = b;
    __syncwarp();
    if (lane == 0) {
      if (rhi > ring_done) psk::st_release_cta_shared_u32(&f->ring_done, rhi);
      if (phi > pool_done) psk::st_release_cta_shared_u32(&f->pool_done, phi);
    }
    if (rhi > ring_done) ring_done = rhi;
    if (phi > pool_done) pool_done = phi;
  }
}

// grid: (slot chunks, instances)
__global__ void __launch_bounds__(kCollectThreads)
leaf_collect_kernel(const uint64_t* __restrict__ slots, const psk::TableDesc* __restrict__ tdesc,
                    const unsigned long long* __restrict__ count, const uint64_t* __restrict__ cap, psk::LruMeta meta,
                    const uint32_t* __restrict__ slow, uint32_t max_use, Leaf* __restrict__ leafbuf,
                    uint32_t* __restrict__ nleaf) {
  const uint32_t i = blockIdx.y;
  if (slow[i] != 1u || count[i] <= cap[i]) return;  // block-uniform
  const psk::TableDesc d = tdesc[i];
  const uint64_t nslots = (uint64_t)d.nbkt * psk::kBucketSlots;
  const uint64_t stride = 4u * (uint64_t)gridDim.x * kCollectThreads;
  // four slots a thread (tables are whole 8-slot buckets); an empty slot's stamp says so unless blocks
  // carry that stamp too, so only leaves' keys are read (8 bytes a slot instead of 12)
  for (uint64_t x = 4u * ((uint64_t)blockIdx.x * kCollectThreads + threadIdx.x); x < nslots; x += stride) {
    const uint4 lu = __ldcs(reinterpret_cast<const uint4*>(meta.last_use + d.base + x));
    const uint4 ch = __ldcs(reinterpret_cast<const uint4*>(meta.children + d.base + x));
    const uint32_t l[4] = {lu.x, lu.y, lu.z, lu.w}, cc[4] = {ch.x, ch.y, ch.z, ch.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (cc[u] != 0u || (l[u] == psk::kNoUse && max_use != psk::kNoUse)) continue;
      const uint64_t s = d.base + x + (uint64_t)u, key = slots[s];
      if (key == psk::kEmpty || key == psk::kTomb) continue;
      const uint32_t at = atomicAdd(nleaf + i, 1u);
      if (at < (uint32_t)kLeafMax)
        leafbuf[(uint64_t)i * kLeafMax + at] = make_leaf(l[u], (uint32_t)s, key, meta.parent[s]);
    }
  }
}

__global__ void __launch_bounds__(kEvictThreads)
evict_kernel(uint64_t* slots, unsigned long long* count, const uint64_t* __restrict__ cap, psk::LruMeta meta,
             const uint32_t* __restrict__ slow, const Leaf* __restrict__ leafbuf, const uint32_t* __restrict__ nleaf,
             uint32_t* more, uint32_t* err) {
  extern __shared__ __align__(16) unsigned char ev_smem[];
  __shared__ EvictFlags flags;
  Leaf* leaves = reinterpret_cast<Leaf*>(ev_smem);
  PoolRec* pool = reinterpret_cast<PoolRec*>(ev_smem + kOffPool);
  ParentRec* ring = reinterpret_cast<ParentRec*>(ev_smem + kOffRing);
  uint32_t* dkey = reinterpret_cast<uint32_t*>(ev_smem + kOffDKey);
  uint32_t* dval = reinterpret_cast<uint32_t*>(ev_smem + kOffDVal);
  Leaf* heap = reinterpret_cast<Leaf*>(ev_smem + kOffHeap);
  const uint32_t i = blockIdx.x;
  const unsigned long long cnt = count[i];
  if (slow[i] != 1u || cnt <= cap[i]) return;  // block-uniform
  // an earlier round gave up: no more rounds (read once, so that the whole block leaves together)
  if (__syncthreads_or(threadIdx.x == 0 && (*(volatile uint32_t*)err & psk::kErrTimeout) != 0u)) return;
  const uint32_t n = nleaf[i];
  if (n > (uint32_t)kLeafMax || n == 0) {
    if (threadIdx.x == 0) atomicOr(err, psk::kErrLeavesFull);
    return;
  }
  uint32_t np2 = 1;
  while (np2 < n) np2 <<= 1;
  for (uint32_t x = threadIdx.x; x < np2; x += kEvictThreads)
    leaves[x] = x < n ? leafbuf[(uint64_t)i * kLeafMax + x]
                      : Leaf{0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, kLeafNoParent};
  __syncthreads();
  for (uint32_t size = 2; size <= np2; size <<= 1) {  // bitonic sort by (last_use, hash)
    for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
      for (uint32_t x = threadIdx.x; x < np2; x += kEvictThreads) {
        const uint32_t y = x ^ stride;
        if (y > x) {
          const bool up = (x & size) == 0;
          const Leaf a = leaves[x], b = leaves[y];
          if (leaf_less(b, a) == up) {
            leaves[x] = b;
            leaves[y] = a;
          }
        }
      }
      __syncthreads();
    }
  }
  const uint64_t E = cnt - cap[i];
  const uint32_t todo = E < (uint64_t)kHeapMax ? (uint32_t)E : (uint32_t)kHeapMax;
  const uint32_t m = n < todo ? n : todo;  // sorted leaves a round can take
  for (uint32_t x = threadIdx.x; x < (uint32_t)kDeltaSlots; x += kEvictThreads) dkey[x] = kLeafNoParent;
  if (threadIdx.x == 0) flags = EvictFlags{0u, 0u, 0u, 0u, 0u};
  __syncthreads();
  const uint32_t warp = threadIdx.x >> 5;
  if (warp >= 2) return;
  if (warp == 1) {
    evict_loader(slots, meta, leaves, ring, pool, m, &flags, err);
  } else if (threadIdx.x == 0) {
    uint32_t ptr = 0, npush = 0;
    int hn = 0;
    uint32_t evicted = 0;
    while (evicted < todo) {
      const bool from_sorted = ptr < n && (hn == 0 || leaf_less(leaves[ptr], heap[0]));
      if (!from_sorted && hn == 0) break;
      Leaf v;
      uint32_t ps = kLeafNoParent;
      ParentRec r{0u, 0u, 0u, 0u, kLeafNoParent};
      if (from_sorted) {
        v = leaves[ptr];
        ps = v.parent;
        if (ps != kLeafNoParent) {
          if (psk::ld_relaxed_cta_shared_u32(&flags.ring_done) > ptr) {
            psk::fence_acq_rel_cta();
            r = ring[ptr % (uint32_t)kRing];
          } else {
            r = load_parent(slots, meta, ps);
          }
        }
        ++ptr;
        psk::st_release_cta_shared_u32(&flags.ptr, ptr);  // the record is read: its slot may be refilled
      } else {
        v = heap_pop(heap, hn);
        if (v.parent != kLeafNoParent) {
          ps = pool[v.parent].pp;
          if (psk::ld_relaxed_cta_shared_u32(&flags.pool_done) > v.parent) {
            psk::fence_acq_rel_cta();
            r = pool[v.parent].r;
          } else {
            r = load_parent(slots, meta, ps);
          }
        }
      }
      slots[v.slot] = psk::kEmpty;
      meta.last_use[v.slot] = psk::kNoUse;
      meta.children[v.slot] = 0;
      meta.parent[v.slot] = psk::kNoParent;
      ++evicted;
      if (ps != kLeafNoParent && count_dec(dkey, dval, ps, r.pc) == 0u) {
        uint32_t link = kLeafNoParent;
        if (r.ppp != kLeafNoParent) {  // ask the loader for the record of its parent
          link = npush;
          pool[npush].pp = r.ppp;
          psk::st_release_cta_shared_u32(&flags.req, ++npush);
        }
        heap_push(heap, hn, Leaf{r.plu, ps, r.ph_lo, r.ph_hi, link});
      }
    }
    count[i] = cnt - evicted;
    if (evicted > 0 && cnt - evicted > cap[i]) atomicOr(more, kMoreSlow);
    psk::st_release_cta_shared_u32(&flags.exit, 1u);
  }
  __syncwarp();
  asm volatile("bar.sync 1, 64;" ::: "memory");  // warps 0 and 1: the loop and the loader are done
  for (uint32_t x = threadIdx.x; x < (uint32_t)kDeltaSlots; x += 64u)
    if (dkey[x] != kLeafNoParent) meta.children[dkey[x]] = dval[x];
}

// Prefix closure check (search mode): every chain's parent must be cached once the chains are in.
__global__ void check_parents_kernel(const uint64_t* slots, const uint64_t* ovf, const psk::TableDesc* __restrict__ tdesc, uint32_t I,
                                     uint64_t nchains, const uint32_t* __restrict__ inst,
                                     const uint64_t* __restrict__ parent, uint32_t* err) {
  for (uint64_t c = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; c < nchains; c += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t p = parent[c];
    const uint32_t i = inst[c];
    if (p == psk::kEmpty || i >= I) continue;
    if (!psk::main_contains(slots, ovf, tdesc[i], p)) atomicOr(err, psk::kErrParentMissing);
  }
}

__global__ void validate_window_kernel(psk::WindowDev w, uint64_t max_blocks, uint32_t* err, unsigned long long* nblk) {
  if (nblk && blockIdx.x == 0 && threadIdx.x == 0) *nblk = w.off[w.R];
  for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < w.R; r += gridDim.x * blockDim.x) {
    const uint64_t a = w.off[r], b = w.off[r + 1];
    const uint32_t L = w.L[r];
    bool ok = b >= a && (b - a) == (uint64_t)(L / 16u) && L < (1u << 30) && b <= max_blocks;
    if (r == 0) ok = ok && a == 0;
    if (!ok) atomicOr(err, psk::kErrWindowLayout);
  }
}

}  // namespace

namespace pskl {

cudaError_t launch_insert_chains(uint64_t* slots, uint64_t* ovf, const psk::TableDesc* tdesc, uint32_t I,
                                 unsigned long long* count, uint64_t nchains, const uint32_t* inst,
                                 const uint64_t* off, const uint64_t* hash, const uint64_t* parent,
                                 uint64_t total, psk::LruMeta meta, uint32_t last_use, uint32_t* err,
                                 int num_sms, cudaStream_t s) {
  if (total == 0 || nchains == 0) return cudaSuccess;
  uint64_t blocks = (nchains + 255) / 256;
  if (blocks > (uint64_t)num_sms * 8) blocks = (uint64_t)num_sms * 8;
  check_instances_kernel<<<(unsigned)blocks, 256, 0, s>>>(I, nchains, inst, err);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(insert_chains_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(InsSmem));
  if (e != cudaSuccess) return e;
  insert_chains_kernel<<<I, kInsThreads, sizeof(InsSmem), s>>>(slots, ovf, tdesc, I, count, nchains, inst, off, hash,
                                                               parent, meta, last_use, err);
  return cudaGetLastError();
}

cudaError_t launch_commit(uint64_t* slots, uint64_t* ovf, const psk::TableDesc* tdesc, uint32_t I,
                          unsigned long long* count, const psk::WindowDev& w, const int32_t* assign,
                          const uint32_t* hit_chosen, psk::LruMeta meta, uint32_t last_use,
                          const psk::ReqStore& rq, const uint32_t* out_tokens, unsigned long long* prefix,
                          uint32_t* err, int num_sms, cudaStream_t s) {
  if (w.R == 0) return cudaSuccess;
  unsigned long long* pre_s = prefix;          // [R + 1]
  unsigned long long* pre_i = prefix + w.R + 1;  // [R + 1]
  commit_prefix_kernel<<<1, 1024, 0, s>>>(w, assign, hit_chosen, pre_s, pre_i);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const uint32_t g = (uint32_t)num_sms * 8u;  // flat items, grid-stride
  if (meta.last_use) {
    commit_stamp_kernel<<<g, 256, 0, s>>>(slots, ovf, tdesc, w, assign, pre_s, meta, last_use);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  commit_insert_kernel<<<g, 256, 0, s>>>(slots, ovf, tdesc, count, w, assign, hit_chosen, pre_i, meta, last_use, err);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (meta.last_use) {
    commit_link_kernel<<<g, 256, 0, s>>>(slots, ovf, tdesc, w, assign, hit_chosen, pre_i, meta);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (rq.M) {
    const uint32_t warps_per_block = 4;
    commit_queue_kernel<<<(I + warps_per_block - 1) / warps_per_block, 32 * warps_per_block, 0, s>>>(
        I, w, assign, hit_chosen, rq, out_tokens, err);
    e = cudaGetLastError();
  }
  return e;
}

cudaError_t launch_advance(psk::StateSoA st, uint32_t I, const psk::ReqStore& rq, const psk::DevModel& m,
                           float window_ms, uint64_t prefill_tokens, uint32_t* err, cudaStream_t s) {
  const uint32_t warps_per_block = 4;
  advance_kernel<<<(I + warps_per_block - 1) / warps_per_block, 32 * warps_per_block, 0, s>>>(
      st, I, rq, m, window_ms, prefill_tokens, err);
  return cudaGetLastError();
}

cudaError_t launch_evict(uint64_t* slots, const psk::TableDesc* tdesc, uint32_t I, unsigned long long* count,
                         const uint64_t* cap, psk::LruMeta meta, EvictScratch& sc, uint32_t* more_host,
                         uint64_t max_instance_slots, uint32_t max_use, uint32_t* err, int num_sms, cudaStream_t s) {
  const size_t smem = kEvictSmem;
  cudaError_t e = cudaFuncSetAttribute(evict_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(evict_order_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(OrderSmem));
  if (e != cudaSuccess) return e;
  EvictPlan* plan = static_cast<EvictPlan*>(sc.plan);
  const uint64_t nb = I < kEvictBatch ? I : kEvictBatch;  // instances a round
  uint32_t* const nlist = sc.list + nb;
  EvictBlocks eb;
  eb.key = static_cast<uint64_t*>(sc.blocks);
  eb.slot = reinterpret_cast<uint32_t*>(eb.key + nb * kClassMax);
  eb.par = eb.slot + nb * 2u * kClassMax;
  eb.jump = reinterpret_cast<uint16_t*>(eb.par + nb * 2u * kClassMax);
  eb.rel = reinterpret_cast<uint8_t*>(eb.jump + nb * kClassMax);
  const uint64_t chunks = (max_instance_slots + kScanChunk - 1) / kScanChunk;
  const unsigned scan_grid = (unsigned)num_sms * 4u;
  const unsigned inst_grid = I < (uint32_t)num_sms ? I : (unsigned)num_sms;
  // histogram passes until a bin is one last_use value
  int passes = 1;
  for (uint64_t v = (uint64_t)max_use >> kHistBits; v; v >>= kHistBits) ++passes;
  const uint64_t per_block = (uint64_t)kCollectThreads * kCollectSlotsPerThread;
  const unsigned gx = (unsigned)((max_instance_slots + per_block - 1) / per_block);
  // The first round launches the kernels that the call before turned out to need: the list says on the device
  // which are needed now, and the others find nothing to do.  Instances left to the one-at-a-time kernels wait
  // for the last batch, and then go together.
  uint32_t todo = sc.class_first ? kMoreFast : kMoreSlow;
  for (int round = 0; round < 4096 && todo; ++round) {
    const bool class_runs = (todo & kMoreFast) != 0u;
    if (class_runs || round == 0) {
      evict_list_kernel<<<1, 1024, 0, s>>>(I, count, cap, sc.slow, sc.nleaf, max_use, plan, sc.list, nlist, sc.more,
                                           round == 0, class_runs);
    } else {
      if ((e = cudaMemsetAsync(sc.more, 0, sizeof(uint32_t), s)) != cudaSuccess) return e;
      if ((e = cudaMemsetAsync(sc.nleaf, 0, (size_t)I * sizeof(uint32_t), s)) != cudaSuccess) return e;
    }
    if (class_runs) {
      for (int pass = 0; pass < passes; ++pass) {
        evict_hist_kernel<<<scan_grid, kScanThreads, 0, s>>>(tdesc, meta, plan, sc.list, nlist, chunks, sc.hist, pass == 0);
        evict_choose_kernel<<<inst_grid, 256, 0, s>>>(plan, sc.list, nlist, sc.hist);
      }
      evict_gather_kernel<<<scan_grid, kScanThreads, 0, s>>>(tdesc, meta, plan, sc.list, nlist, chunks, eb);
      evict_detail_kernel<<<scan_grid, kDetailThreads, 0, s>>>(slots, meta, plan, sc.list, nlist, eb);
      evict_index_kernel<false><<<scan_grid, kDetailThreads, 0, s>>>(meta, plan, sc.list, nlist, kLeafMax, eb);
      evict_index_kernel<true><<<scan_grid, kDetailThreads, 0, s>>>(meta, plan, sc.list, nlist, kLeafMax, eb);
      evict_order_kernel<<<inst_grid, kOrderThreads, sizeof(OrderSmem), s>>>(slots, count, cap, meta, plan, sc.list, nlist,
                                                                            eb, sc.slow, sc.more, kLeafMax, err);
    }
    if (!class_runs) {
      leaf_collect_kernel<<<dim3(gx ? gx : 1u, I), kCollectThreads, 0, s>>>(
          slots, tdesc, count, cap, meta, sc.slow, max_use, static_cast<Leaf*>(sc.leafbuf), sc.nleaf);
      evict_kernel<<<I, kEvictThreads, smem, s>>>(slots, count, cap, meta, sc.slow, static_cast<const Leaf*>(sc.leafbuf),
                                                  sc.nleaf, sc.more, err);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(more_host, sc.more, sizeof(uint32_t), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    if (round == 0) sc.class_first = (*more_host & kMoreListed) != 0u;
    todo = (*more_host & (kMoreFast | kMoreSlow)) | (class_runs ? todo & kMoreSlow : 0u);
  }
  return cudaSuccess;
}

size_t evict_plan_bytes(uint32_t I) { return (size_t)I * sizeof(EvictPlan); }
size_t evict_hist_words(uint32_t I) { return (size_t)(I < kEvictBatch ? I : kEvictBatch) * kHistBins; }
size_t evict_blocks_bytes(uint32_t I) {  // per block: hash, two slots and parents, jump, two relations
  return (size_t)(I < kEvictBatch ? I : kEvictBatch) * kClassMax * (8 + 2 * 4 + 2 * 4 + 2 + 2);
}

size_t evict_leafbuf_bytes(uint32_t I) { return (size_t)I * kLeafMax * sizeof(Leaf); }

cudaError_t launch_check_parents(const uint64_t* slots, const uint64_t* ovf, const psk::TableDesc* tdesc, uint32_t I,
                                 uint64_t nchains, const uint32_t* inst, const uint64_t* parent,
                                 uint32_t* err, int num_sms, cudaStream_t s) {
  if (nchains == 0) return cudaSuccess;
  uint64_t blocks = (nchains + 255) / 256;
  if (blocks > (uint64_t)num_sms * 8) blocks = (uint64_t)num_sms * 8;
  check_parents_kernel<<<(unsigned)blocks, 256, 0, s>>>(slots, ovf, tdesc, I, nchains, inst, parent, err);
  return cudaGetLastError();
}

cudaError_t launch_validate_window(const psk::WindowDev& w, uint64_t max_blocks, uint32_t* err,
                                   unsigned long long* nblk, cudaStream_t s) {
  if (w.R == 0) return cudaSuccess;
  uint32_t blocks = (w.R + 255) / 256;
  if (blocks > 1024) blocks = 1024;
  validate_window_kernel<<<blocks, 256, 0, s>>>(w, max_blocks, err, nblk);
  return cudaGetLastError();
}

}  // namespace pskl
