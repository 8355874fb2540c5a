// Per-request window constants for the greedy pass, computed for all requests in parallel.
//
// Besides the Algorithm 1 / Eq. 8 row constants (T_pf(0, L), CacheBenefit Z, eta * Z, the TTFT
// budget), each request gets its chain relations to earlier requests of the same window:
//   * lcp[d - 1]: the common chain prefix with the request d places before it (d = 1..kLcpBack).  Chained
//     block hashes (Section 7's prefix tree) make "block k equal" imply "blocks 0..k equal", so the
//     common prefix is found with the 32-ary first-miss search.
//   * par: the deepest earlier request whose whole chain is a prefix of this one (an agentic
//     session's previous step, Section 3): its last block equals this chain's block at its length.
//     Its chain end is where this request's hit on the instance that took the parent most likely
//     ends.
//   * anc: the parent's parent and its parent, for the greedy's probe placement.
//   * base: the topmost request reached through par links.  This request's chain starts with the
//     base's whole chain, so on any cache its hit equals the base's hit unless the base is cached
//     in full; the probe derives such rows from the base's row.
// Every hit derived from these relations is exact as far as equal chained hashes mean equal
// prefixes, the same premise as the prefix search of the cached tables.
#include <algorithm>

#include "ps_internal.cuh"

namespace {

constexpr uint32_t kParentScan = 1024;  // chain positions scanned back from the end for a parent (16K tokens)

__device__ __forceinline__ uint32_t tab_home(uint64_t key, uint32_t n) {  // n is a power of two
  return (uint32_t)((key * 0x9E3779B97F4A7C15ull) >> 32) & (n - 1);
}

// Bit of a key in a bit set of `words` (a power of two) words.
__device__ __forceinline__ uint32_t bloom_bit(uint64_t key, uint32_t words) {
  return (uint32_t)((key * 0xD1B54A32D192ED03ull) >> 40) & (words * 32u - 1u);
}
constexpr uint32_t kBloomMaxWords = 8192;  // 2^18 bits, 32 KB of shared memory: 24 key bits suffice

// Table of last-block hashes: each key keeps the earliest request whose chain ends with it.  And the bit
// set of these hashes.
__global__ void lastblock_build_kernel(psk::WindowDev w, psk::LastSlot* tab, uint32_t n, uint32_t* bloom,
                                       uint32_t bloom_words) {
  for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < w.R; r += gridDim.x * blockDim.x) {
    const uint64_t o = w.off[r], nb = w.off[r + 1] - o;
    if (nb == 0) continue;
    const unsigned long long key = w.hash[o + nb - 1];
    if (key == psk::kEmpty || key == psk::kTomb) continue;
    const uint32_t bit = bloom_bit(key, bloom_words);
    atomicOr(bloom + (bit >> 5), 1u << (bit & 31u));
    uint32_t b = tab_home(key, n);
    for (uint32_t p = 0; p < n; ++p) {
      const unsigned long long old = atomicCAS(&tab[b].key, (unsigned long long)psk::kEmpty, key);
      if (old == psk::kEmpty || old == key) {
        atomicMax(&tab[b].neg_idx, 0xFFFFFFFFu - r);
        break;
      }
      b = (b + 1) & (n - 1);
    }
  }
}

// Earliest request whose chain ends with key, -1 if none.  The first slot is loaded by the caller
// (first), so several lookups can be in flight together; collisions continue the linear probe.
__device__ __forceinline__ int32_t tab_resolve(const psk::LastSlot* tab, uint32_t n, uint64_t key, ulonglong2 first) {
  if (key == psk::kEmpty || key == psk::kTomb) return -1;
  uint32_t b = tab_home(key, n);
  ulonglong2 v = first;
  for (uint32_t p = 0; p < n; ++p) {
    if (v.x == key) return (int32_t)(0xFFFFFFFFu - (uint32_t)v.y);
    if (v.x == psk::kEmpty) return -1;
    b = (b + 1) & (n - 1);
    v = __ldg(reinterpret_cast<const ulonglong2*>(tab + b));
  }
  return -1;
}

// Equal blocks that can be cached: a reserved hash says nothing about the prefix it ends.
__device__ __forceinline__ bool same_block(uint64_t x, uint64_t y) { return x == y && x + 1ull > 1ull; }

constexpr int kScanPerLane = 8;  // parent-scan positions per lane and step (256 per warp step)
static_assert(psk::kLcpBack == 32, "one lane per earlier request");

// One warp per request.  Chained block hashes (Section 7's prefix tree) make "block k equal" stand
// for "blocks 0..k equal", as in every prefix search of this library: the common prefix with an
// earlier request is a first-miss search, and an earlier request whose last block equals this
// chain's block at its own length is a prefix of this chain.
//   lcp: lane d holds request r - 1 - d.  Most pairs need no search of their own: the shorter chain is
//        a prefix of the other (a session's earlier step), or the common prefix is the one that other
//        pairs have (the shared system prompt).  So every lane first compares the last common position;
//        then one open pair at a time is searched by the whole warp (32-ary) and every open lane tests
//        that answer on its own pair (two positions), narrowing its range if it fails.  Production
//        window (1024 x 16384): the pass took 0.27 ms for 32 pairs a request, and 0.38 ms for 20 pairs
//        searched four at a time (both before the bit set below).
//   par: the deepest of those requests that is a prefix of this one; if there is none (and the window
//        holds requests before them), the last kParentScan positions are scanned back from the chain's
//        end, 256 per warp step: the deepest position whose block ends an earlier request of exactly
//        that length gives the parent.  A request whose parent lies further back is searched from
//        scratch (exact), and any prefix will do as the parent.  Nearly every scanned block ends no
//        request: a bit set of the last blocks in shared memory (at least 8 bits a request up to 32768
//        requests) sorts those out, so that few lanes read the table (16384 requests: 0.14 ms against 0.22 ms
//        with every position looked up in the table).
__global__ void __launch_bounds__(256, 4)
relations_kernel(psk::WindowDev w, psk::DevModel m, const psk::LastSlot* tab, uint32_t n,
                 const uint32_t* __restrict__ bloom, uint32_t bloom_words, psk::RowPre* rows) {
  extern __shared__ uint32_t s_bloom[];
  const int lane = threadIdx.x & 31;
  const uint32_t wpb = blockDim.x >> 5;
  for (uint32_t x = threadIdx.x; x < bloom_words; x += blockDim.x) s_bloom[x] = bloom[x];
  __syncthreads();
  for (uint32_t r = blockIdx.x * wpb + (threadIdx.x >> 5); r < w.R; r += gridDim.x * wpb) {
    const uint64_t o = w.off[r];
    const uint64_t nb = w.off[r + 1] - o;
    const uint64_t* a = w.hash + o;
    const bool has = r > (uint32_t)lane;  // request q = r - 1 - lane
    uint64_t oq = 0;
    uint32_t nq = 0u;
    if (has) {
      oq = w.off[r - 1 - lane];
      nq = (uint32_t)(w.off[r - lane] - oq);
    }
    const uint64_t* b = w.hash + oq;
    // the first difference lies in [lo, hi] (hi: the end of the shorter chain, or a known difference)
    uint32_t lo = 0u, hi = has ? (uint32_t)(nb < nq ? nb : nq) : 0u;
    if (hi > 0u) {
      if (same_block(a[hi - 1], b[hi - 1])) lo = hi;
      else hi -= 1u;
    }
    for (;;) {
      const unsigned open = __ballot_sync(0xffffffffu, lo < hi);
      if (!open) break;
      const int src = __ffs(open) - 1;
      const uint64_t* bs = w.hash + __shfl_sync(0xffffffffu, oq, src);
      const uint32_t ls = __shfl_sync(0xffffffffu, lo, src), hs = __shfl_sync(0xffffffffu, hi, src);
      const uint32_t x =
          (uint32_t)psk::warp_search_range(ls, hs, [&](uint64_t k) { return same_block(a[k], bs[k]); });
      if (lane == src) {
        lo = hi = x;
      } else if (lo < hi && x >= lo && x <= hi) {  // this pair may well part at x too
        const bool below = x == lo || same_block(a[x - 1], b[x - 1]);
        const bool at = x >= hi || !same_block(a[x], b[x]);
        if (!below) hi = x - 1u;
        else if (at) lo = hi = x;
        else lo = x + 1u;
      }
    }
    const uint32_t lcp = lo;
    const uint32_t hint = __reduce_min_sync(0xffffffffu, has ? lcp : 0xFFFFFFFFu);
    int32_t par = -1;
    uint32_t par_nb = 0;
    {  // the deepest of the last kLcpBack requests whose whole chain is a prefix of this one, latest first
      const uint32_t whole = has && lcp == nq ? nq : 0u;
      const uint32_t best = __reduce_max_sync(0xffffffffu, whole);
      if (best > 0u) {
        par = (int32_t)(r - (uint32_t)__ffs(__ballot_sync(0xffffffffu, whole == best)));
        par_nb = best;
      }
    }
    const uint64_t stop = nb > kParentScan ? nb - kParentScan : 0;
    for (uint64_t top = r > (uint32_t)psk::kLcpBack ? nb : 0; top > stop && par < 0;) {
      const uint64_t lo_s = top - stop > 32u * kScanPerLane ? top - 32u * kScanPerLane : stop;
      uint64_t key[kScanPerLane];
      ulonglong2 first[kScanPerLane];
#pragma unroll
      for (int u = 0; u < kScanPerLane; ++u) {  // position top - 1 - lane - 32 u
        const uint64_t back = (uint64_t)lane + 32u * u;
        key[u] = back < top - lo_s ? a[top - 1 - back] : psk::kEmpty;
      }
#pragma unroll
      for (int u = 0; u < kScanPerLane; ++u) {
        const uint32_t bit = bloom_bit(key[u], bloom_words);
        const bool look = key[u] != psk::kEmpty && key[u] != psk::kTomb && ((s_bloom[bit >> 5] >> (bit & 31u)) & 1u);
        if (!look) key[u] = psk::kEmpty;
        first[u] = look ? __ldg(reinterpret_cast<const ulonglong2*>(tab + tab_home(key[u], n)))
                        : make_ulonglong2(psk::kEmpty, 0ull);
      }
#pragma unroll
      for (int u = 0; u < kScanPerLane; ++u) {
        const uint64_t back = (uint64_t)lane + 32u * u;
        const uint64_t k = top - 1 - back;
        int32_t cand = -1;
        if (key[u] != psk::kEmpty) {
          const int32_t q = tab_resolve(tab, n, key[u], first[u]);
          if (q >= 0 && (uint32_t)q < r && w.off[q + 1] - w.off[q] == k + 1) cand = q;
        }
        const unsigned ok = __ballot_sync(0xffffffffu, cand >= 0);
        if (ok) {  // lower lanes hold deeper positions
          const int src = __ffs(ok) - 1;
          par = __shfl_sync(0xffffffffu, cand, src);
          par_nb = (uint32_t)(top - 32u * u - (uint64_t)src);
          break;
        }
      }
      top = lo_s;
    }
    if (lane == 0) {
      const psk::RowConst rc = psk::row_const(m, w.L[r], w.ttft_t[r], w.tpot_t[r]);
      psk::RowPre x{};
      x.off = o;
      x.nb = (uint32_t)nb;
      x.L = rc.L;
      x.t_cached = rc.t_cached;
      x.c_max = rc.Z > 0.0f ? rc.etaZ : 3.402823466e38f;
      x.tpot_lim = m.slo_off ? INFINITY : rc.tpot_target;
      x.ttft_max = (m.slo_off || !m.ttft_filter) ? INFINITY : rc.ttft_budget;
      x.tpot_target = rc.tpot_target;
      x.hint = r > 0u ? hint : 0u;
      x.limit = (uint32_t)nb;
      x.par = par;
      x.par_nb = par_nb;
      x.base = par;  // base_kernel follows the links from here
      rows[r] = x;
    }
    __syncwarp();
    rows[r].lcp[lane] = lcp;
  }
}

// First reserved hash of each chain (rows' limit), one warp per request.
__global__ void __launch_bounds__(256)
limit_kernel(psk::WindowDev w, psk::RowPre* rows) {
  const uint32_t lane = threadIdx.x & 31u;
  for (uint32_t r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < w.R; r += (gridDim.x * blockDim.x) >> 5) {
    const uint64_t o = w.off[r], nb = w.off[r + 1] - o;
    for (uint64_t k0 = 0; k0 < nb; k0 += 32) {
      const uint64_t key = k0 + lane < nb ? w.hash[o + k0 + lane] : 1ull;
      const unsigned res = __ballot_sync(0xffffffffu, key == psk::kEmpty || key == psk::kTomb);
      if (res) {
        if (lane == 0) rows[r].limit = (uint32_t)k0 + (uint32_t)__ffs(res) - 1u;
        break;
      }
    }
  }
}

// base and the two next ancestors of each request: follow the parent links (parents come
// earlier, so the walk ends).  Requests without a parent go to the list of rows the probe
// searches from scratch.  base starts as par and every walk stores how far it is, so walks through the
// same session shorten one another (a popular session's links run through a thousand requests: 8.5 us
// against 18.7 with each walk on its own, 16384 requests).
__global__ void base_kernel(uint32_t R, psk::RowPre* rows, psk::RowList list) {
  for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < R; r += gridDim.x * blockDim.x) {
    int32_t a = rows[r].par;
    if (a < 0) list.rows[atomicAdd(list.count, 1u)] = r;  // searched from scratch
    int32_t anc[2] = {-1, -1};
    uint32_t anc_nb[2] = {0u, 0u};
    if (a >= 0) {
      anc[0] = rows[a].par;
      if (anc[0] >= 0) {
        anc_nb[0] = rows[a].par_nb;
        anc[1] = rows[anc[0]].par;
        if (anc[1] >= 0) anc_nb[1] = rows[anc[0]].par_nb;
      }
      volatile int32_t* mine = &rows[r].base;
      for (int32_t p = *(volatile int32_t*)&rows[a].base; p >= 0; p = *(volatile int32_t*)&rows[a].base) {
        a = p;
        *mine = a;
      }
    }
    rows[r].base = a;
    rows[r].anc[0] = anc[0];
    rows[r].anc[1] = anc[1];
    rows[r].anc_nb[0] = anc_nb[0];
    rows[r].anc_nb[1] = anc_nb[1];
  }
}

}  // namespace

namespace pskl {

cudaError_t launch_relations(const psk::WindowDev& w, const psk::DevModel& m, psk::LastSlot* tab, uint32_t tab_n,
                             psk::RowPre* rows, psk::RowList list, int search, int num_sms, cudaStream_t s) {
  if (w.R == 0) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  const int g1 = (int)std::min<uint64_t>((w.R + 255) / 256, (uint64_t)num_sms * 8);
  // the table and the bit set behind it, sized by the window; a window of up to kLcpBack + 1 requests
  // needs neither (every earlier request is compared)
  uint32_t n = 0, words = 0;
  uint32_t* bloom = nullptr;
  if (w.R > (uint32_t)psk::kLcpBack + 1u) {
    n = 64;
    while (n < 2u * w.R && n < tab_n) n <<= 1;
    words = std::min(kBloomMaxWords, n / 4u);  // 8 bits a slot, 16 a request
    bloom = reinterpret_cast<uint32_t*>(tab + n);
    e = cudaMemsetAsync(tab, 0, (size_t)n * sizeof(psk::LastSlot) + words * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    lastblock_build_kernel<<<g1, 256, 0, s>>>(w, tab, n, bloom, words);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  // one request per warp: blocks queue, so long rows balance out; with the bit set to load, four blocks
  // an SM that stay
  int g2 = (int)((w.R + 7) / 8);
  const int g3 = words > 256u && g2 > num_sms * 4 ? num_sms * 4 : g2;
  relations_kernel<<<g3, 256, words * sizeof(uint32_t), s>>>(w, m, tab, n, bloom, words, rows);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (!search) limit_kernel<<<g2 < num_sms * 8 ? g2 : num_sms * 8, 256, 0, s>>>(w, rows);
  base_kernel<<<g1, 256, 0, s>>>(w.R, rows, list);
  return cudaGetLastError();
}

}  // namespace pskl
