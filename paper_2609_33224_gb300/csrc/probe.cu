// Probe kernel: prefix-hit length of every (request, instance) pair of a window.
//
// hit(r, i) = the first chain position k whose block hash is not cached on instance i (= the
// chain length if every block is cached): the cached prefix of the request on that instance, the
// quantity the paper's scheduler reads from its prefix tree (Section 7) to estimate KVC reuse.
//
//   linear mode (any cache): a work item is (row, group of instances), one warp per instance, 64
//     consecutive chain positions per step (two lookups per lane in flight), __ballot_sync collecting
//     the misses and __ffs finding the first.
//   search mode (prefix-closed caches, where "block k cached" is monotone along the chain): the
//     rows without an earlier prefix in the window come as a list from the relations pass; a work
//     item is (row, chunk of 256 instances), one lane per instance.  A lane first looks up the
//     row's hint position and the one before it together: the hint is the shortest common prefix
//     with the previous requests of the window, which on most instances is exactly the cached
//     prefix (typically a shared system prompt), so most pairs end after one round trip; the
//     others binary-search the rest of their range.  Without relations (allocation-free scoring)
//     one block takes a request, its chain staged in shared memory, and searches every instance.
//
// Rows whose chain starts with the whole chain of an earlier request of the window (its base, from
// the relations pass) are derived in a second pass instead: the two chains agree block by block up
// to the base's length nb_b, so on any cache hit(r, i) = hit(base, i) when that is below nb_b, and
// otherwise the first miss lies in [nb_b, nb_r) with everything below known cached.  Only those
// instances (the ones caching the base in full) are searched, by a warp each.  Agentic sessions
// resend their history with each step (Section 3), so most rows of a window are derived.
#include "ps_internal.cuh"

namespace {

constexpr uint32_t kStageBlocks = 4096;  // 32 KB of staged chain per thread block

// Launch statistics (ps_last_probe_stats): each warp adds its threads' counts once, at the end.
enum { kStatRowsScratch = 0, kStatRowsDerived, kStatLookupsScratch, kStatLookupsDerived, kStatChainReads,
       kStatPairsDerived };

__device__ __forceinline__ void add_stat(unsigned long long* p, uint64_t v) {
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(p, (unsigned long long)v);
}

// Where a pair's result goes: its hit and, when requested, T_pf at that hit (the greedy pass reads
// it instead of recomputing it for pairs whose hit does not change).
struct PairOut {
  uint32_t* hits;
  float* tpf;
  const uint32_t* L;
  psk::DevModel m;
  __device__ __forceinline__ void put(uint32_t r, uint32_t I, uint32_t i, uint32_t h, uint32_t Lr) const {
    hits[(uint64_t)r * I + i] = h;
    if (tpf) tpf[(uint64_t)r * I + i] = psk::t_pf_of_hit(m, Lr, h);
  }
};

template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32)
probe_hits_kernel(const uint64_t* __restrict__ slots, const uint64_t* __restrict__ ovf,
                  const psk::TableDesc* __restrict__ tdesc,
                  uint32_t I, const uint64_t* __restrict__ off, const uint64_t* __restrict__ hash,
                  uint32_t R, PairOut out) {
  extern __shared__ uint64_t s_chain[];
  for (uint32_t r = blockIdx.x; r < R; r += gridDim.x) {
    const uint64_t o = off[r];
    const uint64_t nb = off[r + 1] - o;
    const uint32_t Lr = out.tpf ? __ldg(out.L + r) : 0u;
    const uint64_t ns = nb < kStageBlocks ? nb : kStageBlocks;
    for (uint64_t k = threadIdx.x; k < ns; k += WARPS * 32) s_chain[k] = __ldg(hash + o + k);
    __syncthreads();
    auto chain = [&](uint64_t k) { return k < ns ? s_chain[k] : __ldg(hash + o + k); };
    for (uint32_t i = threadIdx.x; i < I; i += WARPS * 32) {
      const psk::TableDesc d = tdesc[i];
      uint64_t lo = 0, hi = nb;  // first miss in [lo, hi]
      while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        if (psk::main_contains(slots, ovf, d, chain(mid))) lo = mid + 1; else hi = mid;
      }
      out.put(r, I, i, (uint32_t)lo, Lr);
    }
    __syncthreads();
  }
}

// Linear mode, the rows of the list (or all R rows): see the file comment.  A row's instances are spread
// over the grid: with a block per row (its warps taking the instances in turn, 32 positions a step) 100
// instances x 71 listed rows of about 290 cached blocks took 0.28 ms, 0.073 ms now.
template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32)
probe_linear_kernel(const uint64_t* __restrict__ slots, const uint64_t* __restrict__ ovf,
                    const psk::TableDesc* __restrict__ tdesc, uint32_t I, const uint64_t* __restrict__ off,
                    const uint64_t* __restrict__ hash, uint32_t R, psk::RowList list, PairOut out,
                    unsigned long long* __restrict__ stats) {
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
  const uint32_t ngroup = (I + WARPS - 1) / WARPS;
  const uint64_t items = (uint64_t)(list.rows ? __ldg(list.count) : R) * ngroup;
  uint64_t n_look = 0, n_rows = 0;
  for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const uint32_t r = list.rows ? __ldg(list.rows + item / ngroup) : (uint32_t)(item / ngroup);
    const uint32_t group = (uint32_t)(item % ngroup);
    if (threadIdx.x == 0 && group == 0) n_rows += 1;
    const uint32_t i = group * WARPS + warp;
    if (i >= I) continue;  // warp-uniform
    const uint64_t o = __ldg(off + r);
    const uint64_t nb = __ldg(off + r + 1) - o;
    const uint64_t* chain = hash + o;
    const psk::TableDesc d = tdesc[i];
    uint64_t h = nb;
    for (uint64_t base = 0; base < nb; base += 64) {
      const uint64_t ka = base + lane, kb = ka + 32;
      const uint64_t key_a = ka < nb ? __ldg(chain + ka) : psk::kEmpty, key_b = kb < nb ? __ldg(chain + kb) : psk::kEmpty;
      psk::Lookup la, lb;
      psk::lookup_issue(slots, ovf, d, key_a, la);
      psk::lookup_issue(slots, ovf, d, key_b, lb);
      n_look += (ka < nb ? 1u : 0u) + (kb < nb ? 1u : 0u);
      const bool pa = psk::lookup_finish(slots, ovf, d, key_a, la), pb = psk::lookup_finish(slots, ovf, d, key_b, lb);
      const unsigned ma = __ballot_sync(0xffffffffu, ka < nb && !pa), mb = __ballot_sync(0xffffffffu, kb < nb && !pb);
      if (ma | mb) {
        h = base + (ma ? (uint64_t)(__ffs(ma) - 1) : 32u + (uint64_t)(__ffs(mb) - 1));
        break;
      }
    }
    if (lane == 0) out.put(r, I, i, (uint32_t)h, out.tpf ? __ldg(out.L + r) : 0u);
  }
  if (stats) {
    add_stat(stats + kStatRowsScratch, n_rows);
    add_stat(stats + kStatLookupsScratch, n_look);
    add_stat(stats + kStatChainReads, n_look);
  }
}

// Membership of every lane's key in its instance's table, the buckets read by quads of lanes: a load
// instruction then covers 8 whole buckets (64 bytes by 4 lanes) instead of 16 bytes of 32 buckets, a
// quarter of the lines the L1 looks up (production window, 6.3M lookups: 0.27 ms with a bucket read by
// its own lane, 0.23 ms now; the rest is random access to 0.8 GB of buckets).  All lanes call it.  The first part issues the loads (and, where
// EARLY, the overflow word that only a miss needs), the second compares.
struct QuadLookup {
  ulonglong2 v[8];
  uint64_t ow;
  uint32_t b1;
};

template <bool EARLY>
__device__ __forceinline__ void quad_issue(const uint64_t* __restrict__ slots, const uint64_t* __restrict__ ovf,
                                           const psk::TableDesc& d, uint64_t key, QuadLookup& L) {
  const uint32_t lane = threadIdx.x & 31u;
  L.b1 = psk::fastrange32(key, d.nbkt);
  const uint64_t s1 = d.base + (uint64_t)L.b1 * psk::kBucketSlots;
  const uint64_t s2 = d.base + (uint64_t)psk::fastrange32(psk::remix(key), d.nbkt) * psk::kBucketSlots;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t src = (lane & ~3u) + j;
    const uint64_t a1 = __shfl_sync(0xffffffffu, s1, src), a2 = __shfl_sync(0xffffffffu, s2, src);
    L.v[j] = __ldg(reinterpret_cast<const ulonglong2*>(slots + a1) + (lane & 3u));
    L.v[4 + j] = __ldg(reinterpret_cast<const ulonglong2*>(slots + a2) + (lane & 3u));
  }
  L.ow = EARLY ? __ldg(ovf + d.ovf + (L.b1 >> 6)) : 0ull;
}

template <bool EARLY>
__device__ __forceinline__ bool quad_finish(const uint64_t* __restrict__ slots, const uint64_t* __restrict__ ovf,
                                            const psk::TableDesc& d, uint64_t key, const QuadLookup& L) {
  const uint32_t lane = threadIdx.x & 31u;
  bool hit = false;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint64_t k = __shfl_sync(0xffffffffu, key, (lane & ~3u) + j);
    const bool m = L.v[j].x == k || L.v[j].y == k || L.v[4 + j].x == k || L.v[4 + j].y == k;
    const unsigned b = __ballot_sync(0xffffffffu, m);
    if ((lane & 3u) == (uint32_t)j) hit = (b >> (lane & ~3u)) & 0xFu;
  }
  if (key == psk::kEmpty || key == psk::kTomb) return false;
  if (hit) return true;
  const uint64_t ow = EARLY ? L.ow : __ldg(ovf + d.ovf + (L.b1 >> 6));
  if (!((ow >> (L.b1 & 63u)) & 1ull)) return false;
  return psk::main_contains(slots, ovf, d, key);  // rare: the overflow run after b1
}

// Search mode, rows from the list: see the file comment.  Fewer pairs than the grid has warps (up to
// kWarpPairs a warp) are searched by a warp each instead, 32 positions at once, for the latency: one
// request against 64 instances takes 3 dependent rounds instead of 13 (26 us before, 10 now).
constexpr uint32_t kWarpPairs = 2;

template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32)
probe_search_kernel(const uint64_t* __restrict__ slots, const uint64_t* __restrict__ ovf,
                    const psk::TableDesc* __restrict__ tdesc, uint32_t I, const uint64_t* __restrict__ off,
                    const uint64_t* __restrict__ hash, const psk::RowPre* __restrict__ rows, psk::RowList list,
                    PairOut out, unsigned long long* __restrict__ stats) {
  constexpr uint32_t kChunk = WARPS * 32;
  const uint32_t nrows = __ldg(list.count);
  const uint32_t nchunk = (I + kChunk - 1) / kChunk;
  const uint64_t items = (uint64_t)nrows * nchunk;
  uint64_t n_look = 0, n_rows = 0;
  if ((uint64_t)nrows * I <= (uint64_t)gridDim.x * WARPS * kWarpPairs) {  // grid-uniform
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t pairs = (uint64_t)nrows * I;
    if (blockIdx.x == 0 && threadIdx.x == 0) n_rows = nrows;
    for (uint64_t x = (uint64_t)blockIdx.x * WARPS + (threadIdx.x >> 5); x < pairs; x += (uint64_t)gridDim.x * WARPS) {
      const uint32_t r = __ldg(list.rows + x / I), i = (uint32_t)(x % I);
      const uint64_t o = __ldg(off + r);
      const uint64_t nb = __ldg(off + r + 1) - o;
      const uint64_t* chain = hash + o;
      const psk::TableDesc d = tdesc[i];
      auto cached = [&](uint64_t k) {
        ++n_look;
        return psk::main_contains(slots, ovf, d, __ldg(chain + k));
      };
      const uint64_t h = psk::warp_first_miss_search_hint(0, nb, __ldg(&rows[r].hint), cached);
      if (lane == 0) out.put(r, I, i, (uint32_t)h, out.tpf ? __ldg(out.L + r) : 0u);
    }
  } else {
    for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
      const uint32_t r = __ldg(list.rows + item / nchunk);
      const uint32_t chunk = (uint32_t)(item % nchunk);
      if (threadIdx.x == 0 && chunk == 0) n_rows += 1;
      const uint32_t i = chunk * kChunk + threadIdx.x;
      if (i - (threadIdx.x & 31u) >= I) continue;  // warp-uniform
      const bool live = i < I;
      const uint64_t o = __ldg(off + r);
      const uint64_t nb = __ldg(off + r + 1) - o;
      const uint64_t* chain = hash + o;
      const psk::TableDesc d = tdesc[live ? i : I - 1];
      uint64_t lo = 0, hi = nb;  // the first miss lies in [lo, hi]
      if (nb > 0) {
        const uint64_t hint = __ldg(&rows[r].hint);
        if (hint == 0 || hint >= nb) {
          const uint64_t p = hint == 0 ? 0 : nb - 1;
          const uint64_t k = __ldg(chain + p);
          QuadLookup L;
          quad_issue<true>(slots, ovf, d, k, L);
          n_look += live;
          const bool pr = quad_finish<true>(slots, ovf, d, k, L);
          if (pr) lo = p + 1; else hi = p;
        } else {
          // the hint's block is most likely absent, the one before it present
          const uint64_t k1 = __ldg(chain + hint - 1), k2 = __ldg(chain + hint);
          QuadLookup L1, L2;
          quad_issue<false>(slots, ovf, d, k1, L1);
          quad_issue<true>(slots, ovf, d, k2, L2);
          n_look += 2 * (uint32_t)live;
          const bool p1 = quad_finish<false>(slots, ovf, d, k1, L1);
          const bool p2 = quad_finish<true>(slots, ovf, d, k2, L2);
          if (!p1) hi = hint - 1;
          else if (p2) lo = hint + 1;
          else lo = hi = hint;
        }
      }
      if (!live) continue;
      while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        ++n_look;
        if (psk::main_contains(slots, ovf, d, __ldg(chain + mid))) lo = mid + 1; else hi = mid;
      }
      out.put(r, I, i, (uint32_t)lo, out.tpf ? __ldg(out.L + r) : 0u);
    }
  }
  if (stats) {
    add_stat(stats + kStatRowsScratch, n_rows);
    add_stat(stats + kStatLookupsScratch, n_look);
    add_stat(stats + kStatChainReads, n_look);
  }
}

// Second pass: rows with a base.  One block per row; threads copy the base's hits (four instances at a
// time where rows are 16-byte aligned: VEC) and collect the instances that cache the base in full, then
// warps search those past the base's end, or, when they are many (a base short enough to be cached on
// most instances, such as a bare system prompt), lanes search one each from the row's hint.
template <int WARPS, bool SEARCH, bool VEC>
__global__ void __launch_bounds__(WARPS * 32)
probe_derived_kernel(const uint64_t* __restrict__ slots, const uint64_t* __restrict__ ovf,
                     const psk::TableDesc* __restrict__ tdesc, uint32_t I, const uint64_t* __restrict__ hash,
                     uint32_t R, const psk::RowPre* __restrict__ rows, PairOut out,
                     unsigned long long* __restrict__ stats) {
  extern __shared__ uint32_t s_list[];  // I entries
  __shared__ uint32_t s_n;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  uint64_t n_look = 0, n_rows = 0, n_pairs = 0;
  for (uint32_t r = blockIdx.x; r < R; r += gridDim.x) {
    const int32_t b = __ldg(&rows[r].base);
    if (b < 0) continue;  // block-uniform
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const uint32_t nbb = __ldg(&rows[b].nb);
    const uint32_t nbr = __ldg(&rows[r].nb);
    const uint64_t o = __ldg(&rows[r].off);
    const uint32_t Lr = __ldg(&rows[r].L);
    const uint32_t* hb_row = out.hits + (uint64_t)(uint32_t)b * I;
    const bool open = nbb < nbr;  // instances that cache the base in full are searched past its end
    if (VEC) {
      for (uint32_t i = 4u * threadIdx.x; i < I; i += 4u * WARPS * 32) {
        const uint4 h4 = *reinterpret_cast<const uint4*>(hb_row + i);
        const uint32_t hb[4] = {h4.x, h4.y, h4.z, h4.w};
        *reinterpret_cast<uint4*>(out.hits + (uint64_t)r * I + i) = h4;
        if (out.tpf) {
          float tp[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) tp[k] = psk::t_pf32(out.m, Lr, hb[k]);
          *reinterpret_cast<float4*>(out.tpf + (uint64_t)r * I + i) = make_float4(tp[0], tp[1], tp[2], tp[3]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (open && hb[k] >= nbb) s_list[atomicAdd(&s_n, 1u)] = i + k;
      }
    } else {
      for (uint32_t i = threadIdx.x; i < I; i += WARPS * 32) {
        const uint32_t hb = hb_row[i];
        if (hb < nbb || !open) out.put(r, I, i, hb, Lr);
        else s_list[atomicAdd(&s_n, 1u)] = i;
      }
    }
    __syncthreads();
    const uint32_t n = s_n;
    if (threadIdx.x == 0) {
      n_rows += 1;
      n_pairs += n;
    }
    auto contains = [&](uint32_t i, uint64_t k) {
      ++n_look;
      return psk::main_contains(slots, ovf, tdesc[i], __ldg(hash + o + k));
    };
    if (SEARCH && n > 8u * WARPS) {
      const uint32_t hint = __ldg(&rows[r].hint);
      for (uint32_t x = threadIdx.x; x < n; x += WARPS * 32) {
        const uint32_t i = s_list[x];
        uint32_t lo = nbb, hi = nbr;  // the first miss lies in [lo, hi]
        if (hint > lo && hint < hi) {
          if (!contains(i, hint)) {
            hi = hint;
            if (contains(i, hint - 1)) lo = hint;
            else hi = hint - 1;
          } else {
            lo = hint + 1;
          }
        }
        while (lo < hi) {
          const uint32_t mid = (lo + hi) >> 1;
          if (contains(i, mid)) lo = mid + 1; else hi = mid;
        }
        out.put(r, I, i, lo, Lr);
      }
    } else {
      for (uint32_t x = warp; x < n; x += WARPS) {
        const uint32_t i = s_list[x];
        auto cached = [&](uint64_t k) { return contains(i, k); };
        const uint64_t h = SEARCH ? psk::warp_search_range(nbb, nbr, cached) : psk::warp_first_miss_linear(nbb, nbr, cached);
        if (lane == 0) out.put(r, I, i, (uint32_t)h, Lr);
      }
    }
    __syncthreads();
  }
  if (stats) {
    add_stat(stats + kStatRowsDerived, n_rows);
    add_stat(stats + kStatLookupsDerived, n_look);
    add_stat(stats + kStatChainReads, n_look);
    add_stat(stats + kStatPairsDerived, n_pairs);
  }
}

template <int WARPS>
int max_grid(int num_sms) {
  int per_sm = 0, per_sm2 = 0;
  const int smem = (int)(kStageBlocks * sizeof(uint64_t));
  cudaFuncSetAttribute(probe_hits_kernel<WARPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, probe_hits_kernel<WARPS>, WARPS * 32, smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm2, probe_linear_kernel<WARPS>, WARPS * 32, 0);
  if (per_sm2 < per_sm) per_sm = per_sm2;
  int per_sm3 = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm3, probe_search_kernel<WARPS>, WARPS * 32, 0);
  if (per_sm3 < per_sm) per_sm = per_sm3;
  if (per_sm < 1) per_sm = 1;
  return per_sm * num_sms;
}

}  // namespace

namespace pskl {

int probe_max_grid(uint32_t I, int num_sms) {
  return I >= 64 ? max_grid<8>(num_sms) : max_grid<4>(num_sms);
}

cudaError_t launch_probe(const uint64_t* slots, const uint64_t* ovf, const psk::TableDesc* tdesc, uint32_t I,
                         const psk::WindowDev& w, const psk::RowPre* rows, psk::RowList list, uint32_t* hits,
                         float* tpf, const psk::DevModel& m, int grid, int search, unsigned long long* stats,
                         cudaEvent_t ev_mid, cudaStream_t s) {
  if (w.R == 0) return cudaSuccess;
  const PairOut out{hits, tpf, w.L, m};
  const int g = (int)((uint32_t)grid < w.R ? (uint32_t)grid : w.R);
  // a derived row is a few dependent loads and a copy: more blocks than the search's, to overlap them
  const int g2 = (int)(4u * (uint32_t)grid < w.R ? 4u * (uint32_t)grid : w.R);
  const size_t smem = kStageBlocks * sizeof(uint64_t);
  const size_t smem2 = (size_t)I * sizeof(uint32_t);
  const bool vec = (I & 3u) == 0u && (reinterpret_cast<uintptr_t>(hits) & 15u) == 0u &&
                   (reinterpret_cast<uintptr_t>(tpf) & 15u) == 0u;
#define PS_PROBE(W, S)                                                                                      \
  do {                                                                                                      \
    if (S && rows && list.rows)                                                                             \
      probe_search_kernel<W><<<grid, W * 32, 0, s>>>(slots, ovf, tdesc, I, w.off, w.hash, rows, list, out,   \
                                                     stats);                                                \
    else if (S)                                                                                             \
      probe_hits_kernel<W><<<g, W * 32, smem, s>>>(slots, ovf, tdesc, I, w.off, w.hash, w.R, out);          \
    else                                                                                                    \
      probe_linear_kernel<W><<<grid, W * 32, 0, s>>>(slots, ovf, tdesc, I, w.off, w.hash, w.R,              \
                                                     rows ? list : psk::RowList{nullptr, nullptr}, out, stats); \
    cudaError_t e = cudaGetLastError();                                                                     \
    if (e != cudaSuccess || !rows) return e;                                                                \
    if (ev_mid) cudaEventRecord(ev_mid, s);                                                                 \
    if (w.R == 1) return cudaSuccess; /* no earlier request to derive from */                               \
    (vec ? probe_derived_kernel<W, S, true> : probe_derived_kernel<W, S, false>)<<<g2, W * 32, smem2, s>>>( \
        slots, ovf, tdesc, I, w.hash, w.R, rows, out, stats);                                               \
    return cudaGetLastError();                                                                              \
  } while (0)
  if (I >= 64) {
    if (search) PS_PROBE(8, true);
    PS_PROBE(8, false);
  }
  if (search) PS_PROBE(4, true);
  PS_PROBE(4, false);
#undef PS_PROBE
}

}  // namespace pskl
