// Retrieval paths of the GPU LSM: LOOKUP (§III-D, §IV-B, Fig. 2(b)), COUNT
// (§III-E, §IV-C, Fig. 2(c)) and RANGE (§III-E, §IV-D, Fig. 2(d)).
//
// LOOKUP  searches the full levels from the newest (smallest) to the oldest
//         for the first element whose key is >= q; if that element has key q
//         it decides: regular -> found with its value, tombstone -> absent
//         (and the search stops).  The top of each level's search tree is the
//         level's prefix index, a splitter table of 2^16 .. 2^24 entries
//         (about one per 8 elements): two adjacent loads narrow a search to
//         one bin of about one 32-byte sector, and a short binary search
//         finishes inside it.
//         lookup_direct takes the queries in input order (one thread each);
//         bulk_search takes many of them grouped by key range (the "bulk"
//         alternative of §IV-B): the same search, but neighbouring threads
//         read neighbouring parts of each level; lookup_sorted the same for
//         queries that come sorted by key.
// COUNT   per query and level the window [lower_bound(k1), upper_bound(k2))
//         on the original key; the windows of all levels are then merged on
//         the key, newer level first among equal keys, and a key counts when
//         its first element in that order (its newest version) is regular.
//         This replaces the paper's gather + segmented sort + validation of
//         §IV-C by a per-query multi-way merge of windows that are already
//         sorted; the result is the same count.
// RANGE   the same windows (kept from the count pass), an exclusive scan of
//         the counts into offsets, and a second merge that writes each live
//         (key, value) at its offset, keys ascending within a query (§IV-D).
#include "lsm_device.cuh"

namespace gpulsm {
namespace {

constexpr int kThreads = 256;

// lower_bound of key variable `target` in level l: the level's prefix index
// (a splitter table with about one entry per 8 elements) gives the run of the
// target's bin in two adjacent loads; a short binary search finishes inside.
__device__ __forceinline__ uint32_t level_lower_bound(const LevelSet& ls, int l, uint32_t target) {
  const uint32_t* f = ls.fence[l];
  const int fs = ls.fshift[l];
  const uint32_t bin = fence_bin(target, fs), n = ls.n[l];
  return lower_bound_kv(ls.keys[l], fence_at(f, fs, n, bin), fence_at(f, fs, n, bin + 1), target);
}

// Window [lower_bound(t1), lower_bound(t2)) of level l, t1 <= t2.  A narrow
// interval usually has both bounds in one prefix-index bin: the bin's two
// entries are then loaded once and the second search starts at the first
// bound.
__device__ __forceinline__ uint32_t bin_lower_bound(const uint32_t* a, uint32_t lo, uint32_t hi, uint32_t n, int fs,
                                                    uint32_t target, uint32_t& kv);

__device__ __forceinline__ void level_window(const LevelSet& ls, int l, uint32_t t1, uint32_t t2, uint32_t& lo,
                                             uint32_t& hi) {
  const uint32_t* f = ls.fence[l];
  const int fs = ls.fshift[l];
  const uint32_t n = ls.n[l], b1 = fence_bin(t1, fs), b2 = fence_bin(t2, fs);
  const uint32_t s1 = fence_at(f, fs, n, b1), e1 = fence_at(f, fs, n, b1 + 1);
  const uint32_t s2 = b2 == b1 ? s1 : fence_at(f, fs, n, b2), e2 = b2 == b1 ? e1 : fence_at(f, fs, n, b2 + 1);
  // the two bounds' searches are independent (each bin read in one round trip)
  uint32_t kv;
  lo = bin_lower_bound(ls.keys[l], s1, e1, n, fs, t1, kv);
  hi = bin_lower_bound(ls.keys[l], s2, e2, n, fs, t2, kv);
}

// lower_bound of key variable `target` in a level's n keys `a` (128-byte
// aligned, readable slack after the end), which lies in [lo, hi], target's
// bin at shift fs (elements before lo are below it, elements from hi on
// above); kv: the key variable there when the result is < hi.
// Eight keys are read by two 16-byte loads and searched in registers, one
// round trip instead of a chain of dependent loads: the whole bin if it fits
// from its 16-byte aligned start, else the part where the target is to be
// expected by its place among the bin's key variables.  A bin holds about 8
// elements: a third of the bins fit, and for evenly spread keys the guess is
// off by one or two elements, so that about one bin in thirty is bisected.
// (Bisecting every bin that does not fit: 2^24 lookups in one level of 2^27
// 1121 us, in five levels of 33 million 1361; loading up to 16 keys: 1043 and
// 1116, but 128 small dictionaries' 3.3 million lookups 297 instead of 194.)
// A bin above kCrowded elements holds keys that are not spread, and the guess
// would be one more round trip: it is bisected, like what a guess leaves over
// in one loop for all lanes.  (63 batches of 2^16 keys below 2^16: 2^18 lookups
// 20.5 us bisected, 27.4 with a guess and two loops, now 20.5; a limit of 32
// instead of 64: 1.1 million lookups over bins of 32 and 64 elements on average
// 30 and 40 us, now 26 and 33.)
constexpr uint32_t kCrowded = 64;
__device__ __forceinline__ uint32_t bin_lower_bound(const uint32_t* a, uint32_t lo, uint32_t hi, uint32_t n, int fs,
                                                    uint32_t target, uint32_t& kv) {
  kv = 0;
  uint32_t from = lo, to = hi;  // still to be bisected
  if (hi - lo <= kCrowded) {
    uint32_t a0 = lo & ~3u;
    if (hi > a0 + 8) {
      const uint32_t e = lo + __umulhi(hi - lo, target << (32 - fs));
      a0 = max(a0, (max(e, 2u) - 2u) & ~3u);
    }
    const uint4 x = __ldg(reinterpret_cast<const uint4*>(a + a0)), y = __ldg(reinterpret_cast<const uint4*>(a + a0 + 4));
    uint32_t w[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
    if (n - a0 < 8u) {  // the slack is not part of the order
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (a0 + j >= n) w[j] = 0xFFFFFFFFu;
    }
    uint32_t c = 0;
    kv = w[0];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const bool less = w[j] < target;
      c += less ? 1u : 0u;
      if (j < 7 && less) kv = w[j + 1];
    }
    const bool below = c == 0 && a0 > lo, above = c == 8 && a0 + 8 < hi;
    if (!below && !above) return a0 + c;
    if (below) to = a0;
    if (above) from = a0 + 8;
  }
  const uint32_t pos = lower_bound_kv(a, from, to, target);
  if (pos < hi) kv = __ldg(a + pos);
  return pos;
}

// Lookup of one key over the levels (newest first).  The elements of the
// key, if any, lie in its prefix-index bin [lo, hi) (both status bits of a
// key share its bin).
__device__ __forceinline__ void lookup_one(const LevelSet& ls, uint32_t key, uint32_t& val, uint8_t& found) {
  val = 0;
  found = 0;
  if (key > kMaxUserKey) return;
  for (int l = 0; l < ls.count; ++l) {
    const uint32_t* f = ls.fence[l];
    const int fs = ls.fshift[l];
    const uint32_t n = ls.n[l], bin = fence_bin(key << 1, fs);
    const uint32_t hi = fence_at(f, fs, n, bin + 1);
    uint32_t kv;
    const uint32_t pos = bin_lower_bound(ls.keys[l], fence_at(f, fs, n, bin), hi, n, fs, key << 1, kv);
    if (pos < hi && key_of(kv) == key) {
      if (kv & 1u) {
        found = 1;
        val = __ldg(ls.vals[l] + pos);
      }
      return;
    }
  }
}

__global__ void __launch_bounds__(kThreads) lookup_direct(LevelSet ls, const uint32_t* __restrict__ q, uint64_t nq,
                                                          uint32_t* __restrict__ out_v,
                                                          uint8_t* __restrict__ out_f) {
  for (uint64_t i = blockIdx.x * uint64_t(kThreads) + threadIdx.x; i < nq;
       i += uint64_t(gridDim.x) * kThreads) {
    uint32_t v;
    uint8_t f;
    lookup_one(ls, __ldg(q + i), v, f);
    out_v[i] = v;
    out_f[i] = f;
  }
}

// Many lookups at once (the "bulk" alternative of §IV-B): the same search per
// query, in an order in which neighbouring queries read neighbouring parts
// of every level.  A sort of all queries would cost as much as it saves, and
// its results would have to be scattered; here every query keeps its place in
// its tile, so that all traffic beside the searches is in runs:
//   bulk_tile    per tile of 8192 queries: the keys grouped by 256 equal parts
//                of the key range of the oldest level (in no order within),
//                written to the scratch at the tile's place with the
//                position of each in the tile, and the runs (start, count).
//   bulk_chunks  per part, one CTA: prefix sums of its runs over the tiles,
//                and the first tile of every chunk of kBulkChunk queries.
//   bulk_search  per chunk, one CTA: its keys gathered from the runs, grouped
//                by 2048 finer parts of the range, searched in that order,
//                the results written back to the queries' places in the runs.
//   bulk_untile  per tile: the results put in input order.
// The chunks of one part of the range run at about the same time, so that
// each part of a level and of its prefix index comes from HBM once.  (2^24
// lookups, half of them hits: seven levels of 133 million elements 835 us, one
// level of 2^27 469 us; in input order 2197 and 866.  bulk_search takes 723 and 328
// us of that, bound by its instructions and the latency of the loads between
// them: it issues in two cycles of three, DRAM and L2 are a fifth busy.)
constexpr uint32_t kBulkTile = 8192, kBulkParts = 256, kBulkChunk = 2048, kBulkThreads = 512, kBulkSub = 2048;
constexpr uint32_t kBulkItems = kBulkTile / kBulkThreads;          // per thread of the tile kernels
constexpr uint32_t kBulkChunkItems = kBulkChunk / kBulkThreads;    // per thread of the search

struct BulkScratch {
  uint32_t* key;      // per query, in tile order: its key, then its value
  uint16_t* idx;      // its position in the tile
  uint8_t* found;
  uint32_t* runs;     // [part][tile]: start in the tile, count << 16
  uint32_t* pre;      // [part][tile]: queries of the part in the tiles before
  uint32_t* total;    // per part
  uint2* chunk;       // per chunk: (part << 24) | number of the chunk in its part, first tile
  uint32_t ntiles;
};

// The parts: key variables of [lo, lo + 256 * 2^32 / mul), clamped at both
// ends; the range of the oldest level's populated bins.
struct BulkMap {
  uint32_t lo, mul;
  __device__ __forceinline__ explicit BulkMap(const LevelSet& ls) {
    const int l = ls.count - 1, fs = ls.fshift[l];
    const uint32_t nb = fence_bins(fs), bmin = __ldg(ls.fence[l] + nb + 2), bmax = __ldg(ls.fence[l] + nb + 3);
    lo = bmin << fs;
    mul = max(1u, __float2uint_rd(__fdividef(1099511627776.0f, (float(bmax - bmin) + 1.0f) * float(1u << fs))));
  }
  // part in the high word, place in the part in the low one
  __device__ __forceinline__ uint64_t at(uint32_t key) const {
    const uint32_t kv = key << 1;
    const uint64_t x = uint64_t(max(kv, lo) - lo) * mul;
    return x < (uint64_t(kBulkParts) << 32) ? x : (uint64_t(kBulkParts) << 32) - 1;
  }
};

__global__ void __launch_bounds__(kBulkThreads) bulk_tile(LevelSet ls, const uint32_t* __restrict__ q, uint64_t nq,
                                                          BulkScratch b) {
  __shared__ uint32_t s_key[kBulkTile];
  __shared__ uint16_t s_idx[kBulkTile];
  __shared__ uint32_t s_cnt[kBulkParts], s_start[kBulkParts], s_scan[kBulkThreads / 32];
  const uint32_t tid = threadIdx.x, tile = blockIdx.x;
  const uint64_t t0 = uint64_t(tile) * kBulkTile;
  const uint32_t m = uint32_t(nq - t0 < kBulkTile ? nq - t0 : kBulkTile);
  uint32_t key[kBulkItems], slot[kBulkItems];
#pragma unroll
  for (uint32_t j = 0; j < kBulkItems; ++j)
    if (tid + j * kBulkThreads < m) key[j] = __ldg(q + t0 + tid + j * kBulkThreads);
  if (tid < kBulkParts) s_cnt[tid] = 0u;
  const BulkMap map(ls);
  __syncthreads();
#pragma unroll
  for (uint32_t j = 0; j < kBulkItems; ++j)
    if (tid + j * kBulkThreads < m) slot[j] = atomicAdd(&s_cnt[uint32_t(map.at(key[j]) >> 32)], 1u);
  __syncthreads();
  const uint32_t c = tid < kBulkParts ? s_cnt[tid] : 0u;
  uint32_t all;
  const uint32_t start = block_excl_scan<kBulkThreads>(c, s_scan, all);
  if (tid < kBulkParts) {
    s_start[tid] = start;
    b.runs[tid * b.ntiles + tile] = start | (c << 16);
    if (c) atomicAdd(b.total + tid, c);
  }
  __syncthreads();
#pragma unroll
  for (uint32_t j = 0; j < kBulkItems; ++j) {
    if (tid + j * kBulkThreads < m) {
      const uint32_t pos = s_start[uint32_t(map.at(key[j]) >> 32)] + slot[j];
      s_key[pos] = key[j];
      s_idx[pos] = uint16_t(tid + j * kBulkThreads);
    }
  }
  __syncthreads();
  for (uint32_t i = tid; i < m; i += kBulkThreads) {
    b.key[t0 + i] = s_key[i];
    b.idx[t0 + i] = s_idx[i];
  }
}

__device__ __forceinline__ uint32_t bulk_chunks_of(uint32_t total) { return (total + kBulkChunk - 1) / kBulkChunk; }

__global__ void __launch_bounds__(kBulkThreads) bulk_chunks(BulkScratch b) {
  __shared__ uint32_t s_scan[kBulkThreads / 32];
  const uint32_t tid = threadIdx.x, d = blockIdx.x;
  uint32_t base, carry = 0;  // the part's first chunk
  block_excl_scan<kBulkThreads>(tid < d ? bulk_chunks_of(b.total[tid]) : 0u, s_scan, base);
  for (uint32_t t0 = 0; t0 < b.ntiles; t0 += kBulkThreads) {
    const uint32_t t = t0 + tid;
    const uint32_t c = t < b.ntiles ? b.runs[d * b.ntiles + t] >> 16 : 0u;
    uint32_t all;
    const uint32_t before = carry + block_excl_scan<kBulkThreads>(c, s_scan, all);
    if (t < b.ntiles) {
      b.pre[d * b.ntiles + t] = before;
      // the chunks whose first query lies in this run
      for (uint32_t k = (before + kBulkChunk - 1) / kBulkChunk; k * kBulkChunk < before + c; ++k)
        b.chunk[base + k] = make_uint2((d << 24) | k, t);
    }
    carry += all;
  }
}

__global__ void __launch_bounds__(kBulkThreads, 4) bulk_search(LevelSet ls, BulkScratch b) {
  __shared__ uint32_t s_key[kBulkChunk];
  __shared__ uint32_t s_cnt[kBulkSub];     // the finer parts' counters, then the values
  __shared__ uint16_t s_ord[kBulkChunk];
  __shared__ uint8_t s_found[kBulkChunk];
  __shared__ uint32_t s_pre[kBulkThreads], s_base[kBulkThreads], s_scan[kBulkThreads / 32];
  __shared__ uint32_t s_m;
  static_assert(kBulkSub == kBulkChunk, "the values take the counters' place");
  const uint32_t tid = threadIdx.x;
  uint32_t chunks;
  block_excl_scan<kBulkThreads>(tid < kBulkParts ? bulk_chunks_of(b.total[tid]) : 0u, s_scan, chunks);
  if (blockIdx.x >= chunks) return;
  const uint2 desc = b.chunk[blockIdx.x];
  const uint32_t d = desc.x >> 24, first = (desc.x & 0xFFFFFFu) * kBulkChunk;
  const uint32_t last = min(first + kBulkChunk, b.total[d]);
  const BulkMap map(ls);
  uint32_t o = first;
  for (uint32_t t0 = desc.y; o < last; t0 += kBulkThreads) {  // once, unless most tiles have no run of the part
    const uint32_t t = t0 + tid;
    const uint32_t pre = t < b.ntiles ? b.pre[d * b.ntiles + t] : last;
    const uint32_t run = t < b.ntiles ? b.runs[d * b.ntiles + t] : 0u;
    s_pre[tid] = pre;
    s_base[tid] = t * kBulkTile + (run & 0xFFFFu) - pre;
    for (uint32_t i = tid; i < kBulkSub; i += kBulkThreads) s_cnt[i] = 0u;
    if (tid == kBulkThreads - 1) s_m = min(pre + (run >> 16), last);
    __syncthreads();
    const uint32_t m = s_m - o;  // queries [o, o + m) of the part lie in these tiles
    uint32_t at[kBulkChunkItems], key[kBulkChunkItems], sub[kBulkChunkItems];
#pragma unroll
    for (uint32_t j = 0; j < kBulkChunkItems; ++j) {
      const uint32_t i = tid + j * kBulkThreads;
      if (i < m) {
        uint32_t lo = 0, hi = kBulkThreads - 1;  // the largest run with pre <= o + i
        while (lo < hi) {
          const uint32_t mid = (lo + hi + 1) >> 1;
          if (s_pre[mid] <= o + i) lo = mid; else hi = mid - 1;
        }
        at[j] = s_base[lo] + o + i;
        key[j] = b.key[at[j]];
      }
    }
#pragma unroll
    for (uint32_t j = 0; j < kBulkChunkItems; ++j) {
      if (tid + j * kBulkThreads < m) {
        const uint32_t s = uint32_t(map.at(key[j])) / (0xFFFFFFFFu / kBulkSub + 1u);
        sub[j] = s | (atomicAdd(&s_cnt[s], 1u) << 16);
      }
    }
    __syncthreads();
    constexpr uint32_t kPer = kBulkSub / kBulkThreads;
    uint32_t c[kPer], sum = 0;
#pragma unroll
    for (uint32_t e = 0; e < kPer; ++e) {
      c[e] = s_cnt[tid * kPer + e];
      sum += c[e];
    }
    uint32_t all;
    uint32_t runsum = block_excl_scan<kBulkThreads>(sum, s_scan, all);
#pragma unroll
    for (uint32_t e = 0; e < kPer; ++e) {
      s_cnt[tid * kPer + e] = runsum;
      runsum += c[e];
    }
    __syncthreads();
#pragma unroll
    for (uint32_t j = 0; j < kBulkChunkItems; ++j) {
      const uint32_t i = tid + j * kBulkThreads;
      if (i < m) {
        const uint32_t pos = s_cnt[sub[j] & 0xFFFFu] + (sub[j] >> 16);
        s_key[pos] = key[j];
        s_ord[pos] = uint16_t(i);
      }
    }
    __syncthreads();
    for (uint32_t x = tid; x < m; x += kBulkThreads) {
      uint32_t v;
      uint8_t f;
      lookup_one(ls, s_key[x], v, f);
      s_cnt[s_ord[x]] = v;
      s_found[s_ord[x]] = f;
    }
    __syncthreads();
#pragma unroll
    for (uint32_t j = 0; j < kBulkChunkItems; ++j) {
      const uint32_t i = tid + j * kBulkThreads;
      if (i < m) {
        b.key[at[j]] = s_cnt[i];
        b.found[at[j]] = s_found[i];
      }
    }
    o += m;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kBulkThreads) bulk_untile(BulkScratch b, uint64_t nq, uint32_t* __restrict__ val,
                                                            uint8_t* __restrict__ found) {
  __shared__ uint32_t s_val[kBulkTile];
  __shared__ uint8_t s_found[kBulkTile];
  const uint32_t tid = threadIdx.x;
  const uint64_t t0 = uint64_t(blockIdx.x) * kBulkTile;
  const uint32_t m = uint32_t(nq - t0 < kBulkTile ? nq - t0 : kBulkTile);
#pragma unroll 8
  for (uint32_t i = tid; i < m; i += kBulkThreads) {
    const uint32_t x = b.idx[t0 + i];
    s_val[x] = b.key[t0 + i];
    s_found[x] = b.found[t0 + i];
  }
  __syncthreads();
  for (uint32_t i = tid; i < m; i += kBulkThreads) {
    val[t0 + i] = s_val[i];
    found[t0 + i] = s_found[i];
  }
}

// Queries sorted by key: the same per-query search as lookup_direct, in key
// order, so neighbouring threads read neighbouring parts of every level and
// prefix index (few pages and sectors per warp); results scattered back to
// positions idx[i].
__global__ void __launch_bounds__(kThreads) lookup_sorted(LevelSet ls, const uint32_t* __restrict__ sq,
                                                          const uint32_t* __restrict__ idx, uint64_t nq,
                                                          uint32_t* __restrict__ out_v,
                                                          uint8_t* __restrict__ out_f) {
  for (uint64_t i = blockIdx.x * uint64_t(kThreads) + threadIdx.x; i < nq;
       i += uint64_t(gridDim.x) * kThreads) {
    uint32_t v;
    uint8_t f;
    lookup_one(ls, __ldg(sq + i), v, f);
    const uint32_t o = __ldg(idx + i);
    if (o < nq) {  // a permutation of [0, nq) unless the sort gave up on a wait
      out_v[o] = v;
      out_f[o] = f;
    }
  }
}

// Per-query multi-way merge of the level windows on the key, newer level
// first among equal keys; visits the newest element of every key once.  L is
// a compile-time bound on the number of full levels (loops fully unrolled, so
// the cursors stay in registers); levels l >= ls.count are empty.  Once a
// key's newest element is taken, every level skips the whole run of that key
// (a binary search when the run is longer than one element), so keys stored
// many times (stale versions, a short batch's padding) cost O(L log run).
template <bool kEmit, int L>
__device__ __forceinline__ uint32_t merge_windows(const LevelSet& ls, const uint32_t (&lo)[L],
                                                  const uint32_t (&hi)[L], uint32_t* out_k, uint32_t* out_v,
                                                  uint64_t room) {
  if (L == 1 && ls.count == 1 && hi[0] - (lo[0] & ~3u) <= 16) {
    // One level and a short window: its keys (and values) from the 16-byte
    // aligned start in four 16-byte loads each, walked in registers; a key's
    // first element is its newest (level order), kept when regular.
    const uint32_t* a = ls.keys[0];
    const uint32_t a0 = lo[0] & ~3u;
    uint32_t w[16], v[16];
#pragma unroll
    for (int c4 = 0; c4 < 4; ++c4) {
      const uint4 x = __ldg(reinterpret_cast<const uint4*>(a + a0) + c4);
      w[4 * c4] = x.x;
      w[4 * c4 + 1] = x.y;
      w[4 * c4 + 2] = x.z;
      w[4 * c4 + 3] = x.w;
      if (kEmit) {
        const uint4 y = __ldg(reinterpret_cast<const uint4*>(ls.vals[0] + a0) + c4);
        v[4 * c4] = y.x;
        v[4 * c4 + 1] = y.y;
        v[4 * c4 + 2] = y.z;
        v[4 * c4 + 3] = y.w;
      }
    }
    uint32_t c = 0, prev = 0xFFFFFFFFu;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const uint32_t pos = a0 + j;
      if (pos >= lo[0] && pos < hi[0]) {
        const uint32_t k = key_of(w[j]);
        if (k != prev && (w[j] & 1u)) {
          if (kEmit && c < room) {
            out_k[c] = k;
            out_v[c] = v[j];
          }
          ++c;
        }
        prev = k;
      }
    }
    return c;
  }
  uint32_t cur[L], head[L];
#pragma unroll
  for (int l = 0; l < L; ++l) {
    cur[l] = lo[l];
    head[l] = (l < ls.count && cur[l] < hi[l]) ? key_of(__ldg(ls.keys[l] + cur[l])) : 0xFFFFFFFFu;
  }
  uint32_t c = 0;
  while (true) {
    uint32_t bk = 0xFFFFFFFFu, p = 0;
    int best = -1;
#pragma unroll
    for (int l = 0; l < L; ++l)
      if (head[l] < bk) {  // strict: the lowest (newest) level wins ties
        bk = head[l];
        best = l;
        p = cur[l];
      }
    if (best < 0) break;
    const uint32_t kv = __ldg(ls.keys[best] + p);
    if (kv & 1u) {
      if (kEmit && c < room) {
        out_k[c] = bk;
        out_v[c] = __ldg(ls.vals[best] + p);
      }
      ++c;
    }
#pragma unroll
    for (int l = 0; l < L; ++l) {
      if (head[l] == bk) {  // past every element of key bk in level l
        const uint32_t* a = ls.keys[l];
        uint32_t q = cur[l] + 1;
        uint32_t nk = q < hi[l] ? key_of(__ldg(a + q)) : 0xFFFFFFFFu;
        if (nk == bk) {
          q = upper_bound_key(a, q + 1, hi[l], bk);
          nk = q < hi[l] ? key_of(__ldg(a + q)) : 0xFFFFFFFFu;
        }
        cur[l] = q;
        head[l] = nk;
      }
    }
  }
  return c;
}

// With `perm` (queries sorted by k1: k1 holds the sorted lower bounds and
// perm their positions), thread i serves query perm[i] and stores its count
// and windows at that position; neighbouring threads then search
// neighbouring parts of every level.
// Queries whose windows hold more than kWideMin elements in all are wide:
// with a wide list, the count kernel appends them to it (their count and
// output are then written by the warp kernels below) instead of merging
// hundreds of elements in one thread.  (The line comes from the warp kernels'
// first form.  2^18 counts in six levels, windows of 30 / 60 / 90 elements: 305 /
// 341 / 378 us with a line at 16, 142 / 361 / 378 at 40, 138 / 225 / 314 at 120.)
constexpr uint32_t kWideMin = 40;

template <int L>
__device__ __forceinline__ uint32_t window_total(const uint32_t (&lo)[L], const uint32_t (&hi)[L]) {
  uint32_t t = 0;
#pragma unroll
  for (int l = 0; l < L; ++l) t += hi[l] - lo[l];
  return t;
}

template <int L>
__global__ void __launch_bounds__(kThreads) count_kernel(LevelSet ls, const uint32_t* __restrict__ k1,
                                                         const uint32_t* __restrict__ k2, uint64_t nq,
                                                         uint32_t* __restrict__ out_count,
                                                         uint32_t* __restrict__ bounds,
                                                         const uint32_t* __restrict__ perm,
                                                         uint32_t* __restrict__ wide) {
  for (uint64_t i0 = blockIdx.x * uint64_t(kThreads) + threadIdx.x; i0 < nq;
       i0 += uint64_t(gridDim.x) * kThreads) {
    const uint64_t i = perm ? __ldg(perm + i0) : i0;
    if (i >= nq) continue;  // a permutation of [0, nq) unless its sort gave up on a wait
    const uint32_t a = __ldg(k1 + i0);
    uint32_t z = __ldg(k2 + i);
    if (z > kMaxUserKey) z = kMaxUserKey;
    uint32_t lo[L], hi[L];
    const bool empty = a > z;
#pragma unroll
    for (int l = 0; l < L; ++l) {
      lo[l] = hi[l] = 0;
      if (l < ls.count && !empty) level_window(ls, l, a << 1, (z + 1u) << 1, lo[l], hi[l]);
    }
    if (wide && window_total(lo, hi) > kWideMin) {
      wide[1 + atomicAdd(wide, 1u)] = uint32_t(i0);
    } else {
      out_count[i] = merge_windows<false, L>(ls, lo, hi, nullptr, nullptr, 0);
    }
    if (bounds) {
      uint32_t* b = bounds + i * 2 * ls.count;
#pragma unroll
      for (int l = 0; l < L; ++l)
        if (l < ls.count) {
          b[2 * l] = lo[l];
          b[2 * l + 1] = hi[l];
        }
    }
  }
}

template <int L>
__global__ void __launch_bounds__(kThreads) range_emit(LevelSet ls, uint64_t nq,
                                                       const uint32_t* __restrict__ bounds,
                                                       const uint64_t* __restrict__ offsets,
                                                       uint32_t* __restrict__ keys,
                                                       uint32_t* __restrict__ vals,
                                                       const uint32_t* __restrict__ perm, bool wide) {
  for (uint64_t i0 = blockIdx.x * uint64_t(kThreads) + threadIdx.x; i0 < nq;
       i0 += uint64_t(gridDim.x) * kThreads) {
    const uint64_t i = perm ? __ldg(perm + i0) : i0;
    if (i >= nq) continue;
    uint32_t lo[L], hi[L];
    const uint32_t* b = bounds + i * 2 * ls.count;
#pragma unroll
    for (int l = 0; l < L; ++l) {
      lo[l] = l < ls.count ? b[2 * l] : 0u;
      hi[l] = l < ls.count ? b[2 * l + 1] : 0u;
    }
    if (wide && window_total(lo, hi) > kWideMin) continue;  // emitted by range_wide
    const uint64_t o = offsets[i];
    merge_windows<true, L>(ls, lo, hi, keys + o, vals + o, offsets[i + 1] - o);
  }
}

// Wide queries, one warp each.  The warp stages the windows of all levels,
// newest level first, in shared memory (coalesced reads, all in flight).
// Every element then looks for its key in the windows of the older levels:
// levels double, so that these searches are few (each element once per older
// level: about as many as elements in all), while looking from the old
// levels, which hold most elements, into the newer ones takes some four times
// as many.  An element found has a newer version and loses its status bit; what
// is still regular, and the first of its key in its level, is live.  For the
// output order the same searches give every element's place in the merged
// order: c elements of the older level come before the one that searches, and
// that one comes before the older level's elements from c on (a histogram of
// c, summed up).  The places of the live elements are marked in a bitmap
// whose prefix counts give the output positions.
// Windows above kWideCap elements in all are taken in pieces: the keys below
// the smallest of the levels' (kWideCap / levels)-th keys, which at most
// kWideCap elements have; a key that fills a level's share alone is decided by
// itself.
// (2 10^5 queries of about 107 elements in six levels, count_wide + range_wide:
// one lane per 1/32 of the key interval, merging its own windows step by step,
// 618 + 1151 us; searches into the newer levels 499 + 748; this 258 +
// 365 us.  Bound by its instructions.)
constexpr uint32_t kWideCap = 512, kPlaceBits = 9;
static_assert(kWideCap == 1u << kPlaceBits && kMaxLevels <= 64, "a place and its level fit 16 bits");
struct WideCount {
  uint32_t kv[kWideCap];
};
struct WideEmit {
  uint32_t kv[kWideCap], hist[kWideCap];
  uint16_t place[kWideCap];
  uint32_t bits[kWideCap / 32], before[kWideCap / 32];
};

// First of the n elements of the sorted run a whose key variable is >= x.
__device__ __forceinline__ uint32_t lower_bound_smem(const uint32_t* a, uint32_t n, uint32_t x) {
  uint32_t lo = 0;
  while (n) {
    const uint32_t h = n >> 1;
    const bool less = a[lo + h] < x;
    lo = less ? lo + h + 1 : lo;
    n = less ? n - h - 1 : h;
  }
  return lo;
}

// Windows in which most keys repeat (many stale versions in each level): the
// versions are skipped instead of read.  A group of lanes, one per level, takes
// the keys of its part of the windows one after another: the smallest head
// among the lanes is the next key, the newest level's element decides, and
// every lane whose head it is goes to the end of its run, whose length is
// guessed from the run before.  The parts are cut at even places of the largest
// window.  The live keys as wide_merge in x, the number of runs in y; kEmit: the
// parts' counts come from a first pass.  Bound by the chain of loads, a few per
// key and level.
template <bool kEmit, bool kOne>
__device__ __forceinline__ uint2 repeat_merge(const LevelSet& ls, uint32_t pos, uint32_t end, uint32_t* out_k,
                                              uint32_t* out_v, uint64_t room) {
  const uint32_t lane = lane_id();
  uint32_t width = 1;  // lanes of a group
  if (!kOne)
    while (width < uint32_t(ls.count)) width *= 2;
  const uint32_t l = lane & (width - 1), part = lane / width, parts = 32 / width;
  const bool act = l < uint32_t(ls.count);
  const uint32_t *keys = act ? ls.keys[l] : nullptr, *vals = act ? ls.vals[l] : nullptr;
  // the part's start in every level, and the next part's
  const uint32_t most = __reduce_max_sync(0xffffffffu, end - pos);
  const int big = kOne ? 0 : __ffs(int(__ballot_sync(0xffffffffu, end - pos == most))) - 1;
  const uint32_t cut = __shfl_sync(0xffffffffu, pos, big) + uint32_t(uint64_t(most) * part / parts);
  const uint32_t from = part ? key_of(__ldg(ls.keys[big] + cut)) : 0u;
  const uint32_t p = __shfl_sync(0xffffffffu, pos, int(l)), e = __shfl_sync(0xffffffffu, end, int(l));
  const uint32_t start = act ? (part ? lower_bound_kv(keys, p, e, from << 1) : p) : 0u;
  const uint32_t next = __shfl_down_sync(0xffffffffu, start, width);
  const uint32_t stop = act ? (part + 1 < parts ? next : e) : 0u;
  uint32_t before = 0, live = 0, runs = 0;
#pragma unroll 1
  for (int pass = kEmit ? 0 : 1; pass < 2; ++pass) {
    uint32_t cur = start, run = 1;
    uint32_t kv = cur < stop ? __ldg(keys + cur) : 0xFFFFFFFFu;
    uint32_t value = 0, *to_value = nullptr;  // of the last key emitted: stored with the next one
    live = runs = 0;
    for (;;) {
      const uint32_t head = cur < stop ? key_of(kv) : 0xFFFFFFFFu;
      uint32_t k = head;
      for (uint32_t o = 1; o < width; o <<= 1) k = min(k, __shfl_xor_sync(0xffffffffu, k, int(o)));
      if (!__any_sync(0xffffffffu, k != 0xFFFFFFFFu)) break;
      const bool mine = head == k && k != 0xFFFFFFFFu;
      const uint32_t who = __ballot_sync(0xffffffffu, mine), live_who = __ballot_sync(0xffffffffu, mine && (kv & 1u));
      const uint32_t group = who & (0xffffffffu >> (32 - width)) << (part * width);
      const uint32_t newest = group & (0u - group);  // its lane's bit
      if (live_who & newest) {
        if (kEmit && pass && newest == 1u << lane && before + live < room) {
          out_k[before + live] = k;
          if (to_value) *to_value = value;
          to_value = out_v + before + live;
          value = __ldg(vals + cur);
        }
        ++live;
      }
      if (mine) {  // past the run: [cur, at] are of it, kv becomes the element at `to`, which is not
        uint32_t at = cur, to = cur + run;
        for (; to < stop; run *= 2) {
          kv = __ldg(keys + to);
          if (key_of(kv) != k) break;
          at = to;
          to += run;
        }
        to = min(to, stop);
        while (to - at > 1) {
          const uint32_t mid = at + (to - at) / 2, x = __ldg(keys + mid);
          if (key_of(x) == k) {
            at = mid;
          } else {
            to = mid;
            kv = x;
          }
        }
        run = to - cur;
        cur = to;
        ++runs;
      }
    }
    if (to_value) *to_value = value;
    const uint32_t share = l == 0 ? live : 0u;
    const uint32_t sum = warp_incl_scan(share);
    before = __shfl_sync(0xffffffffu, sum - share, int(part * width));
    live = __shfl_sync(0xffffffffu, sum, 31);
  }
  return make_uint2(live, warp_sum(runs));
}

// Versions are skipped from kAgain pieces in a row on that repeat: kSame of 32
// elements have the key of the one before, or a key fills a piece alone.  The
// next kReach elements are then taken by repeat_merge, then four times as many,
// while they have kRepeats per run; when they do not, it takes twice as many
// pieces to come back to it.  One level, which is read straight through, from
// kAgainOne chunks of 128 in a row on that end in 32 of one key (one that is all
// one key counts twice), while there are kRepeatsOne per run.
// (31 batches of 2^18 keys below 2^16, about 24 copies of a key per level:
// 65536 counts of 64 keys 4690 us read piece by piece, so 579, ranges 16.1 and 2.6
// ms; 256 counts of 50000 keys 225 and 19 ms.  One level of 2^24 with 256 copies:
// 65536 counts of 64 keys 1315 and 329 us.  Zipf keys have such pieces, but seldom
// two in a row: 8192 ranges of 1000 keys 430 us read, 434 so, 690 when one piece
// was enough.  range_wide takes 64 registers instead of 48 for it, without which
// the value of a key found is waited for; no fewer CTAs fit beside its shared
// memory.)
constexpr uint32_t kSame = 24, kAgain = 2, kRepeats = 3, kReach = 2048, kMaxReach = 1u << 24;
constexpr uint32_t kAgainOne = 4, kRepeatsOne = 32;

// Live keys of the window [i0, last) of the only level: nothing to look for in
// other levels, so the window is read through, in order.
template <bool kEmit>
__device__ __forceinline__ uint32_t wide_one(const LevelSet& ls, uint32_t i0, const uint32_t last, uint32_t* out_k,
                                             uint32_t* out_v, uint64_t room) {
  const uint32_t lane = lane_id(), lt = lanemask_lt();
  const uint32_t* keys = ls.keys[0];
  uint32_t done = 0, again = 0, before = 0xFFFFFFFFu;  // before: key before the chunk
  while (i0 < last) {
    uint32_t kv[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t i = i0 + 32 * j + lane;
      kv[j] = i < last ? __ldg(keys + i) : 0xFFFFFFFEu;  // (no regular element)
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t k = key_of(kv[j]), up = __shfl_up_sync(0xffffffffu, k, 1);
      const bool ok = (kv[j] & 1u) && k != (lane ? up : before);
      before = __shfl_sync(0xffffffffu, k, 31);
      const uint32_t m = __ballot_sync(0xffffffffu, ok), at = done + __popc(m & lt);
      if (kEmit && ok && at < room) {
        out_k[at] = k;
        out_v[at] = __ldg(ls.vals[0] + (i0 + 32 * j + lane));
      }
      done += __popc(m);
    }
    i0 += 128;
    const bool one = __shfl_sync(0xffffffffu, key_of(kv[0]), 0) == before;
    again = __shfl_sync(0xffffffffu, key_of(kv[3]), 0) == before ? again + (one ? 2u : 1u) : 0u;
    if (i0 >= last || (!one && again < kAgainOne)) continue;
    i0 = upper_bound_key(keys, i0, last, before);  // past a long run (a short batch's padding is one)
    if (again < kAgainOne) continue;
    bool paid = true;
    for (uint32_t reach = kReach; paid && i0 < last; reach = min(4 * reach, kMaxReach)) {
      uint32_t to = last;
      if (last - i0 > reach) {  // up to the start of a run, or the end of one that is longer
        const uint32_t k = key_of(__ldg(keys + i0 + reach));
        to = lower_bound_kv(keys, i0, i0 + reach, k << 1);
        if (to == i0) to = upper_bound_key(keys, i0 + reach, last, k);
      }
      const uint2 got = repeat_merge<kEmit, true>(ls, lane ? 0u : i0, lane ? 0u : to, out_k + done, out_v + done,
                                                  room > done ? room - done : 0u);
      done += got.x;
      paid = to - i0 >= kRepeatsOne * got.y;
      i0 = to;
    }
    again = 0;
    before = 0xFFFFFFFFu;
  }
  return done;
}

// Live keys of the windows [pos, end) (lane l holds level l's) of several
// levels, emitted to out_k/out_v in key order when kEmit (at most `room`);
// returns their number.
template <class Shared>
__device__ __forceinline__ uint32_t wide_merge(const LevelSet& ls, uint32_t pos, uint32_t end, Shared& sh,
                                               uint32_t* out_k, uint32_t* out_v, uint64_t room) {
  constexpr bool kEmit = sizeof(Shared) == sizeof(WideEmit);
  const uint32_t lane = lane_id();
  const int nl = ls.count;
  const bool act = lane < uint32_t(nl);
  const uint32_t* keys = act ? ls.keys[lane] : nullptr;
  uint32_t done = 0, again = 0, enough = kAgain;
  uint32_t reach = 0;  // elements that repeat_merge takes next, 0 when it does not
  for (;;) {
    const uint32_t left = act ? end - pos : 0u;
    const uint32_t total = warp_sum(left);
    if (total == 0) return done;
    // this piece: [pos, pos + n) of every level
    uint32_t n = left;
    const uint32_t cap = max(reach, kWideCap);
    if (total > cap) {
      const uint32_t share = cap / uint32_t(nl);
      const uint32_t lim = __reduce_min_sync(0xffffffffu, left > share ? key_of(__ldg(keys + pos + share)) : 0xFFFFFFFFu);
      n = left ? lower_bound_kv(keys, pos, pos + min(left, share), lim << 1) - pos : 0u;
      if (!__any_sync(0xffffffffu, n != 0u)) {
        // every next element has a key >= lim, and one level starts with more
        // than its share of copies of it
        const uint32_t first = left ? __ldg(keys + pos) : 0xFFFFFFFFu;
        const uint32_t has = __ballot_sync(0xffffffffu, left && key_of(first) == lim);
        const int newest = __ffs(int(has)) - 1;
        const bool live = (__shfl_sync(0xffffffffu, first, newest) & 1u) != 0u;
        if (live) {
          if (kEmit && int(lane) == newest && done < room) {
            out_k[done] = lim;
            out_v[done] = __ldg(ls.vals[lane] + pos);
          }
          ++done;
        }
        if (left && key_of(first) == lim) pos = upper_bound_key(keys, pos, end, lim);
        if (reach) reach = min(4 * reach, kMaxReach);
        else if (++again >= enough) reach = kReach;
        continue;
      }
    }
    if (reach) {
      const uint2 got = repeat_merge<kEmit, false>(ls, pos, pos + n, out_k + done, out_v + done,
                                                   room > done ? room - done : 0u);
      done += got.x;
      pos += n;
      again = 0;
      const bool paid = warp_sum(n) >= kRepeats * got.y;
      if (!paid) enough *= 2;
      reach = paid ? min(4 * reach, kMaxReach) : 0u;
      continue;
    }
    const uint32_t off = warp_incl_scan(n) - n;
    __syncwarp();
    for (int l = 0; l < nl; ++l) {
      const uint32_t m = __shfl_sync(0xffffffffu, n, l), o = __shfl_sync(0xffffffffu, off, l),
                     p = __shfl_sync(0xffffffffu, pos, l);
      const uint32_t* from = ls.keys[l] + p;
      for (uint32_t i = lane; i < m; i += 32) {
        cp_async4(sh.kv + o + i, from + i);
        if constexpr (kEmit) {
          sh.hist[o + i] = 0u;
          sh.place[o + i] = uint16_t(l << kPlaceBits);
        }
      }
    }
    const uint32_t all = warp_sum(n);
    if constexpr (kEmit) {
      if (lane < kWideCap / 32) sh.bits[lane] = 0u;
    }
    cp_async_wait_all();
    __syncwarp();
    for (int l = 1; l < nl; ++l) {  // the elements of the newer levels, [0, o), look into level l
      const uint32_t m = __shfl_sync(0xffffffffu, n, l), o = __shfl_sync(0xffffffffu, off, l);
      if (m == 0) continue;
      for (uint32_t t = lane; t < o; t += 32) {
        const uint32_t x = sh.kv[t] & ~1u, c = lower_bound_smem(sh.kv + o, m, x);
        if (c < m) {
          if ((sh.kv[o + c] & ~1u) == x) sh.kv[o + c] = x;  // (the key and the order stay)
          if constexpr (kEmit) atomicAdd(&sh.hist[o + c], 1u);
        }
        if constexpr (kEmit) sh.place[t] += uint16_t(c);     // this lane's alone; the sum is below kWideCap
      }
    }
    __syncwarp();
    uint32_t live = 0;
    if constexpr (!kEmit) {
      // (at a level's start the element before is a newer level's: one with
      // the same key has taken the status bit)
      for (uint32_t t = lane; t < all; t += 32)
        live += (sh.kv[t] & 1u) && (t == 0 || key_of(sh.kv[t - 1]) != key_of(sh.kv[t])) ? 1u : 0u;
      live = warp_sum(live);
    } else {
      uint32_t sum = 0;
      for (uint32_t t0 = 0; t0 < all; t0 += 32) {  // running sums of the histogram, over all levels
        const uint32_t t = t0 + lane;
        const uint32_t h = sum + warp_incl_scan(t < all ? sh.hist[t] : 0u);
        if (t < all) sh.hist[t] = h;
        sum = __shfl_sync(0xffffffffu, h, 31);
      }
      __syncwarp();
      for (uint32_t t0 = 0; t0 < all; t0 += 32) {
        const uint32_t t = t0 + lane;
        const uint32_t own = t < all ? sh.place[t] : 0u, l = own >> kPlaceBits;
        const uint32_t o = __shfl_sync(0xffffffffu, off, int(l));  // the level's first element here
        if (t < all) {
          const bool ok = (sh.kv[t] & 1u) && (t == 0 || key_of(sh.kv[t - 1]) != key_of(sh.kv[t]));
          const uint32_t place = t - o + (own & (kWideCap - 1)) + sh.hist[t] - (o ? sh.hist[o - 1] : 0u);
          sh.place[t] = ok ? uint16_t((l << kPlaceBits) | place) : uint16_t(0xFFFFu);
          if (ok) atomicOr(&sh.bits[place >> 5], 1u << (place & 31u));
        }
      }
      __syncwarp();
      const uint32_t b = lane < kWideCap / 32 ? uint32_t(__popc(sh.bits[lane])) : 0u;
      const uint32_t incl = warp_incl_scan(b);
      if (lane < kWideCap / 32) sh.before[lane] = incl - b;
      live = __shfl_sync(0xffffffffu, incl, 31);
      __syncwarp();
      for (uint32_t t0 = 0; t0 < all; t0 += 32) {
        const uint32_t t = t0 + lane;
        const uint32_t own = t < all ? sh.place[t] : 0xFFFFu, l = own == 0xFFFFu ? 0u : own >> kPlaceBits;
        const uint32_t from = __shfl_sync(0xffffffffu, pos - off, int(l));  // (may wrap)
        if (own == 0xFFFFu) continue;
        const uint32_t place = own & (kWideCap - 1), w = place >> 5;
        const uint32_t at = done + sh.before[w] + __popc(sh.bits[w] & ((1u << (place & 31u)) - 1u));
        if (at < room) {
          out_k[at] = key_of(sh.kv[t]);
          out_v[at] = __ldg(ls.vals[l] + (from + t));
        }
      }
    }
    done += live;
    pos += n;
    if (total > all) {
      const uint32_t t = 1 + (lane * all) / 33;  // (all > 1: a piece with nothing in it takes a key alone)
      const bool same = t < all && key_of(sh.kv[t - 1]) == key_of(sh.kv[t]);
      again = uint32_t(__popc(__ballot_sync(0xffffffffu, same))) >= kSame ? again + 1 : 0u;
      if (again >= enough) reach = kReach;
    }
  }
}

template <bool kOne>
__global__ void __launch_bounds__(kThreads, 8) count_wide(LevelSet ls, const uint32_t* __restrict__ k1,
                                                          const uint32_t* __restrict__ k2, uint64_t nq,
                                                          uint32_t* __restrict__ out_count,
                                                          const uint32_t* __restrict__ perm,
                                                          const uint32_t* __restrict__ wide) {
  const uint32_t nw = *reinterpret_cast<const volatile uint32_t*>(wide);
  const uint32_t lane = lane_id();
  for (uint32_t w = (blockIdx.x * kThreads + threadIdx.x) >> 5; w < nw; w += (gridDim.x * kThreads) >> 5) {
    const uint32_t i0 = wide[1 + w];
    const uint64_t i = perm ? __ldg(perm + i0) : i0;
    if (i >= nq) continue;  // whole warp
    const uint32_t a = __ldg(k1 + i0), z = min(__ldg(k2 + i), kMaxUserKey);
    uint32_t lo = 0, hi = 0;
    if (lane < uint32_t(ls.count) && a <= z) level_window(ls, int(lane), a << 1, (z + 1u) << 1, lo, hi);
    uint32_t c;
    if constexpr (kOne) {
      c = wide_one<false>(ls, __shfl_sync(0xffffffffu, lo, 0), __shfl_sync(0xffffffffu, hi, 0), nullptr, nullptr, 0);
    } else {
      __shared__ WideCount s_warp[kThreads / 32];
      c = wide_merge(ls, lo, hi, s_warp[threadIdx.x >> 5], nullptr, nullptr, 0);
    }
    if (lane == 0) out_count[i] = c;
  }
}

// The windows are those that the count pass stored.
template <bool kOne>
__global__ void __launch_bounds__(kThreads) range_wide(LevelSet ls, uint64_t nq, const uint32_t* __restrict__ bounds,
                                                          const uint64_t* __restrict__ offsets,
                                                          uint32_t* __restrict__ keys, uint32_t* __restrict__ vals,
                                                          const uint32_t* __restrict__ perm,
                                                          const uint32_t* __restrict__ wide) {
  const uint32_t nw = *reinterpret_cast<const volatile uint32_t*>(wide);
  const uint32_t lane = lane_id();
  for (uint32_t w = (blockIdx.x * kThreads + threadIdx.x) >> 5; w < nw; w += (gridDim.x * kThreads) >> 5) {
    const uint32_t i0 = wide[1 + w];
    const uint64_t i = perm ? __ldg(perm + i0) : i0;
    if (i >= nq) continue;  // whole warp
    uint32_t lo = 0, hi = 0;
    if (lane < uint32_t(ls.count)) {
      lo = __ldg(bounds + (i * ls.count + lane) * 2);
      hi = __ldg(bounds + (i * ls.count + lane) * 2 + 1);
    }
    const uint64_t o = offsets[i], room = offsets[i + 1] - o;
    if constexpr (kOne) {
      wide_one<true>(ls, __shfl_sync(0xffffffffu, lo, 0), __shfl_sync(0xffffffffu, hi, 0), keys + o, vals + o, room);
    } else {
      __shared__ WideEmit s_warp[kThreads / 32];
      wide_merge(ls, lo, hi, s_warp[threadIdx.x >> 5], keys + o, vals + o, room);
    }
  }
}

// SUCCESSOR / PREDECESSOR (the order-based queries the problem statement's
// footnote names beside the three retrievals, read inclusively): the live
// pair with the smallest key >= q, or the largest key <= q.  Each level's
// cursor starts at q's position; the levels are merged on the key from q
// outwards (ascending for the successor, descending for the predecessor),
// newest level first among equal keys; the first key whose newest element is
// regular is the answer, every other key is skipped in all levels at once.
// Within a level a key's newest element is the first of its run, so the
// descending merge looks up each run's start.
template <int L, bool kSucc>
__global__ void __launch_bounds__(kThreads) neighbor_kernel(LevelSet ls, const uint32_t* __restrict__ q,
                                                            uint64_t nq, uint32_t* __restrict__ out_k,
                                                            uint32_t* __restrict__ out_v,
                                                            uint8_t* __restrict__ out_f) {
  for (uint64_t i = blockIdx.x * uint64_t(kThreads) + threadIdx.x; i < nq; i += uint64_t(gridDim.x) * kThreads) {
    const uint32_t key = __ldg(q + i);
    uint32_t rk = 0, rv = 0;
    uint8_t rf = 0;
    uint32_t cur[L], head[L];
    bool live[L];  // the level still has a candidate on the search side
#pragma unroll
    for (int l = 0; l < L; ++l) {
      cur[l] = 0;
      head[l] = 0;
      live[l] = false;
      if (l < ls.count) {
        if (kSucc) {
          if (key <= kMaxUserKey) {
            cur[l] = level_lower_bound(ls, l, key << 1);
            live[l] = cur[l] < ls.n[l];
          }
        } else {
          const uint32_t kq = key < kMaxUserKey ? key : kMaxUserKey;
          const uint32_t e = level_lower_bound(ls, l, (kq + 1u) << 1);  // first key > kq
          live[l] = e > 0;
          cur[l] = live[l] ? e - 1 : 0u;
        }
        if (live[l]) head[l] = key_of(__ldg(ls.keys[l] + cur[l]));
      }
    }
    while (true) {
      int best = -1;
      uint32_t bk = 0;
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!live[l]) continue;
        const bool better = best < 0 || (kSucc ? head[l] < bk : head[l] > bk);  // strict: newest level wins ties
        if (better) {
          bk = head[l];
          best = l;
        }
      }
      if (best < 0) break;
      // newest element of key bk: the run start in the newest level holding it
      uint32_t p = cur[best];
      if (!kSucc) p = lower_bound_kv(ls.keys[best], 0, cur[best] + 1, bk << 1);
      const uint32_t kv = __ldg(ls.keys[best] + p);
      if (kv & 1u) {
        rk = bk;
        rv = __ldg(ls.vals[best] + p);
        rf = 1;
        break;
      }
      // skip key bk in every level
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!live[l] || head[l] != bk) continue;
        const uint32_t* a = ls.keys[l];
        if (kSucc) {
          uint32_t nx = cur[l] + 1;
          if (nx < ls.n[l] && key_of(__ldg(a + nx)) == bk) nx = upper_bound_key(a, nx + 1, ls.n[l], bk);
          cur[l] = nx;
          live[l] = nx < ls.n[l];
          if (live[l]) head[l] = key_of(__ldg(a + nx));
        } else {
          const uint32_t st = lower_bound_kv(a, 0, cur[l] + 1, bk << 1);  // run start of bk
          live[l] = st > 0;
          if (live[l]) {
            cur[l] = st - 1;
            head[l] = key_of(__ldg(a + cur[l]));
          }
        }
      }
    }
    out_k[i] = rk;
    out_v[i] = rv;
    out_f[i] = rf;
  }
}

constexpr int kScanIPT = 8;
constexpr int kScanTile = kThreads * kScanIPT;  // 2048
constexpr uint64_t kLbAgg = 1ull << 62, kLbIncl = 2ull << 62, kLbMask = (1ull << 62) - 1;

__global__ void __launch_bounds__(kThreads) scan_kernel(const uint32_t* __restrict__ in, uint64_t n,
                                                        uint64_t* __restrict__ out, uint64_t* lookback,
                                                        uint32_t* tile_ctr, uint32_t* status,
                                                        uint64_t ntiles) {
  __shared__ uint64_t s_scan[kThreads / 32];
  __shared__ uint64_t s_prefix;
  __shared__ uint32_t s_tile;
  const uint32_t tid = threadIdx.x;
  if (tid == 0) s_tile = atomicAdd(tile_ctr, 1u);
  __syncthreads();
  const uint64_t tile = s_tile;
  const uint64_t base = tile * kScanTile + uint64_t(tid) * kScanIPT;
  uint32_t v[kScanIPT];
  uint64_t sum = 0;
#pragma unroll
  for (int j = 0; j < kScanIPT; ++j) {
    v[j] = base + j < n ? __ldg(in + base + j) : 0u;
    sum += v[j];
  }
  uint64_t tile_sum;
  const uint64_t before = block_excl_scan<kThreads, uint64_t>(sum, s_scan, tile_sum);
  if (tid == 0) {
    uint64_t prefix = 0;
    if (tile == 0) {
      st_relaxed_u64(lookback, kLbIncl | tile_sum);
    } else {
      st_relaxed_u64(lookback + tile, kLbAgg | tile_sum);
      int64_t t = int64_t(tile) - 1;
      uint64_t t0 = 0;
      while (t >= 0) {
        const uint64_t w = ld_relaxed_u64(lookback + t);
        if (!(w & (kLbAgg | kLbIncl))) {
          if (!spin_continue(t0, kWaitLimitNs, status)) break;
          continue;
        }
        prefix += w & kLbMask;
        if (w & kLbIncl) break;
        --t;
      }
      st_relaxed_u64(lookback + tile, kLbIncl | (prefix + tile_sum));
    }
    s_prefix = prefix;
    if (tile == ntiles - 1) out[n] = prefix + tile_sum;
  }
  __syncthreads();
  uint64_t run = s_prefix + before;
#pragma unroll
  for (int j = 0; j < kScanIPT; ++j) {
    if (base + j < n) out[base + j] = run;
    run += v[j];
  }
}

unsigned persistent_grid(uint64_t work, int per_block, unsigned cap) {
  uint64_t b = (work + per_block - 1) / per_block;
  if (b > cap) b = cap;
  return unsigned(b ? b : 1);
}

// Lookup in the batched form: query g belongs to instance i with
// qoff[i] <= g < qoff[i + 1] and searches that instance's full levels (the
// set bits of r_i), newest first, exactly as lookup_one does.
__global__ void __launch_bounds__(kThreads) multi_lookup(MultiArena ar, const uint32_t* __restrict__ q,
                                                         const uint64_t* __restrict__ qoff, uint64_t nq,
                                                         uint32_t* __restrict__ out_v,
                                                         uint8_t* __restrict__ out_f) {
  for (uint64_t g = blockIdx.x * uint64_t(kThreads) + threadIdx.x; g < nq; g += uint64_t(gridDim.x) * kThreads) {
    const uint32_t i = find_instance(qoff, ar.n, g);
    const MultiInst& d = ar.inst[i];
    const uint32_t key = __ldg(q + g);
    uint32_t val = 0;
    uint8_t found = 0;
    if (key <= kMaxUserKey) {
      uint32_t r = ar.r[i];
      while (r) {
        const int l = __ffs(r) - 1;
        r &= r - 1;
        const uint32_t* keys = ar.keys + d.lvl_off[l];
        const uint32_t* f = ar.fence + d.lvl_fence[l];
        const int fs = d.lvl_fshift[l];
        const uint32_t n = d.b << l, bin = fence_bin(key << 1, fs);
        const uint32_t hi = fence_at(f, fs, n, bin + 1);
        uint32_t kv;
        const uint32_t pos = bin_lower_bound(keys, fence_at(f, fs, n, bin), hi, n, fs, key << 1, kv);
        if (pos < hi && key_of(kv) == key) {
          if (kv & 1u) {
            found = 1;
            val = __ldg(ar.vals + d.lvl_off[l] + pos);
          }
          break;
        }
      }
    }
    out_v[g] = val;
    out_f[g] = found;
  }
}

}  // namespace

cudaError_t lookup_launch(const LevelSet& ls, const uint32_t* q, uint64_t nq, uint32_t* val, uint8_t* found,
                          cudaStream_t st) {
  if (nq == 0) return cudaSuccess;
  count_launches(1);
  lookup_direct<<<persistent_grid(nq, kThreads, 152 * 8), kThreads, 0, st>>>(ls, q, nq, val, found);
  return cudaGetLastError();
}

static BulkScratch bulk_scratch(void* p, uint64_t nq) {
  BulkScratch b{};
  b.ntiles = uint32_t((nq + kBulkTile - 1) / kBulkTile);
  const uint64_t padded = uint64_t(b.ntiles) * kBulkTile;
  b.key = static_cast<uint32_t*>(p);
  b.runs = b.key + padded;
  b.pre = b.runs + uint64_t(kBulkParts) * b.ntiles;
  b.chunk = reinterpret_cast<uint2*>(b.pre + uint64_t(kBulkParts) * b.ntiles);
  b.total = reinterpret_cast<uint32_t*>(b.chunk + padded / kBulkChunk + kBulkParts);
  b.idx = reinterpret_cast<uint16_t*>(b.total + kBulkParts);
  b.found = reinterpret_cast<uint8_t*>(b.idx + padded);
  return b;
}

size_t lookup_bulk_bytes(uint64_t nq) {
  const BulkScratch b = bulk_scratch(nullptr, nq);
  return size_t(reinterpret_cast<uintptr_t>(b.found)) + size_t(b.ntiles) * kBulkTile;
}

cudaError_t lookup_bulk_launch(const LevelSet& ls, const uint32_t* q, uint64_t nq, uint32_t* val, uint8_t* found,
                               void* scratch, cudaStream_t st) {
  if (nq == 0) return cudaSuccess;
  const BulkScratch b = bulk_scratch(scratch, nq);
  cudaError_t e = cudaMemsetAsync(b.total, 0, kBulkParts * sizeof(uint32_t), st);
  if (e != cudaSuccess) return e;
  count_launches(4);
  bulk_tile<<<b.ntiles, kBulkThreads, 0, st>>>(ls, q, nq, b);
  bulk_chunks<<<kBulkParts, kBulkThreads, 0, st>>>(b);
  bulk_search<<<unsigned((nq + kBulkChunk - 1) / kBulkChunk + kBulkParts), kBulkThreads, 0, st>>>(ls, b);
  bulk_untile<<<b.ntiles, kBulkThreads, 0, st>>>(b, nq, val, found);
  return cudaGetLastError();
}

cudaError_t lookup_sorted_launch(const LevelSet& ls, const uint32_t* sq, const uint32_t* idx, uint64_t nq,
                                 uint32_t* val, uint8_t* found, cudaStream_t st) {
  if (nq == 0) return cudaSuccess;
  count_launches(1);
  lookup_sorted<<<persistent_grid(nq, kThreads, 152 * 8), kThreads, 0, st>>>(ls, sq, idx, nq, val, found);
  return cudaGetLastError();
}

cudaError_t count_launch(const LevelSet& ls, const uint32_t* k1, const uint32_t* k2, uint64_t nq,
                         uint32_t* count, uint32_t* bounds, cudaStream_t st, const uint32_t* perm,
                         uint32_t* wide) {
  if (nq == 0) return cudaSuccess;
  cudaError_t e;
  if (wide && (e = cudaMemsetAsync(wide, 0, sizeof(uint32_t), st)) != cudaSuccess) return e;
  const unsigned grid = persistent_grid(nq, kThreads, 152 * 8);
  count_launches(1);
  if (ls.count <= 1) count_kernel<1><<<grid, kThreads, 0, st>>>(ls, k1, k2, nq, count, bounds, perm, wide);
  else if (ls.count <= 2) count_kernel<2><<<grid, kThreads, 0, st>>>(ls, k1, k2, nq, count, bounds, perm, wide);
  else if (ls.count <= 4) count_kernel<4><<<grid, kThreads, 0, st>>>(ls, k1, k2, nq, count, bounds, perm, wide);
  else if (ls.count <= 8) count_kernel<8><<<grid, kThreads, 0, st>>>(ls, k1, k2, nq, count, bounds, perm, wide);
  else if (ls.count <= 16) count_kernel<16><<<grid, kThreads, 0, st>>>(ls, k1, k2, nq, count, bounds, perm, wide);
  else count_kernel<kMaxLevels><<<grid, kThreads, 0, st>>>(ls, k1, k2, nq, count, bounds, perm, wide);
  if ((e = cudaGetLastError()) != cudaSuccess || !wide) return e;
  // the wide queries, one warp each (the grid covers every query's warp when
  // all are wide; an empty list ends at once)
  const unsigned wgrid = persistent_grid(nq * 32, kThreads, 152 * 8);
  count_launches(1);
  if (ls.count <= 1) count_wide<true><<<wgrid, kThreads, 0, st>>>(ls, k1, k2, nq, count, perm, wide);
  else count_wide<false><<<wgrid, kThreads, 0, st>>>(ls, k1, k2, nq, count, perm, wide);
  return cudaGetLastError();
}

cudaError_t scan_launch(const uint32_t* in, uint64_t n, uint64_t* out, uint64_t* lookback, uint32_t* tile_ctr,
                        uint32_t* status, cudaStream_t st) {
  cudaError_t e;
  if (n == 0) return cudaMemsetAsync(out, 0, sizeof(uint64_t), st);
  const uint64_t ntiles = scan_tiles(n);
  if ((e = cudaMemsetAsync(lookback, 0, sizeof(uint64_t) * ntiles, st)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(tile_ctr, 0, sizeof(uint32_t), st)) != cudaSuccess) return e;
  count_launches(1);
  scan_kernel<<<unsigned(ntiles), kThreads, 0, st>>>(in, n, out, lookback, tile_ctr, status, ntiles);
  return cudaGetLastError();
}

cudaError_t range_emit_launch(const LevelSet& ls, uint64_t nq, const uint32_t* bounds, const uint64_t* offsets,
                              uint32_t* keys, uint32_t* vals, cudaStream_t st, const uint32_t* perm,
                              const uint32_t* wide) {
  if (nq == 0) return cudaSuccess;
  cudaError_t e;
  const bool w = wide != nullptr;
  const unsigned grid = persistent_grid(nq, kThreads, 152 * 8);
  count_launches(1);
  if (ls.count <= 1) range_emit<1><<<grid, kThreads, 0, st>>>(ls, nq, bounds, offsets, keys, vals, perm, w);
  else if (ls.count <= 2) range_emit<2><<<grid, kThreads, 0, st>>>(ls, nq, bounds, offsets, keys, vals, perm, w);
  else if (ls.count <= 4) range_emit<4><<<grid, kThreads, 0, st>>>(ls, nq, bounds, offsets, keys, vals, perm, w);
  else if (ls.count <= 8) range_emit<8><<<grid, kThreads, 0, st>>>(ls, nq, bounds, offsets, keys, vals, perm, w);
  else if (ls.count <= 16) range_emit<16><<<grid, kThreads, 0, st>>>(ls, nq, bounds, offsets, keys, vals, perm, w);
  else range_emit<kMaxLevels><<<grid, kThreads, 0, st>>>(ls, nq, bounds, offsets, keys, vals, perm, w);
  if ((e = cudaGetLastError()) != cudaSuccess || !w) return e;
  const unsigned wgrid = persistent_grid(nq * 32, kThreads, 152 * 8);
  count_launches(1);
  if (ls.count <= 1) range_wide<true><<<wgrid, kThreads, 0, st>>>(ls, nq, bounds, offsets, keys, vals, perm, wide);
  else range_wide<false><<<wgrid, kThreads, 0, st>>>(ls, nq, bounds, offsets, keys, vals, perm, wide);
  return cudaGetLastError();
}


cudaError_t multi_lookup_launch(const MultiArena& ar, const uint32_t* q, const uint64_t* qoff, uint64_t nq,
                                uint32_t* val, uint8_t* found, cudaStream_t st) {
  if (nq == 0) return cudaSuccess;
  count_launches(1);
  multi_lookup<<<persistent_grid(nq, kThreads, 152 * 8), kThreads, 0, st>>>(ar, q, qoff, nq, val, found);
  return cudaGetLastError();
}


cudaError_t neighbor_launch(const LevelSet& ls, const uint32_t* q, uint64_t nq, bool successor, uint32_t* key,
                            uint32_t* val, uint8_t* found, cudaStream_t st) {
  if (nq == 0) return cudaSuccess;
  const unsigned grid = persistent_grid(nq, kThreads, 152 * 8);
  count_launches(1);
#define LSM_NB(LL)                                                                                   \
  (successor ? (neighbor_kernel<LL, true><<<grid, kThreads, 0, st>>>(ls, q, nq, key, val, found), 0) \
             : (neighbor_kernel<LL, false><<<grid, kThreads, 0, st>>>(ls, q, nq, key, val, found), 0))
  if (ls.count <= 1) LSM_NB(1);
  else if (ls.count <= 2) LSM_NB(2);
  else if (ls.count <= 4) LSM_NB(4);
  else if (ls.count <= 8) LSM_NB(8);
  else if (ls.count <= 16) LSM_NB(16);
  else LSM_NB(kMaxLevels);
#undef LSM_NB
  return cudaGetLastError();
}

}  // namespace gpulsm
