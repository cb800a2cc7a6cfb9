// Batch sort of the GPU LSM: a stable radix sort of (key variable, value) pairs
// over all 32 bits (§IV-A sorts every batch with a radix sort over the whole
// key variable, status bit included, so a tombstone precedes a regular element
// of the same key).  Up to 5120 elements one CTA sorts the batch (small_sort),
// up to 2^20 msd_tile and bucket_sort do, whose comments are further down; what
// follows is the least-significant-digit sort above that, 8 bits per pass.
//
// Structure (one histogram kernel, then one kernel per digit):
//   * sort_histogram reads the input once and counts all four digits; in the
//     batch modes it also encodes each op as (key << 1) | status and checks
//     that keys are below 2^31 - 1.
//   * sort_pass ranks a tile of 8192 elements per CTA in shared memory, gets
//     the tile's global offset per digit from the tiles before it by
//     decoupled look-back (tile order comes from an atomic ticket, so a CTA
//     only ever waits on CTAs that already started), and scatters.
// In the batch modes the first pass reads the input back to front, padded at
// the logical end with copies of the last op; a stable sort of that sequence
// puts the last of several equal key variables first (the "last insert wins"
// reading of §III-A rule 4).
#include "lsm_device.cuh"
#include "sort_maps.h"

namespace gpulsm {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kRadix = 256;
constexpr uint32_t kNoDigit = 256;
// A pass: 512 threads of 16 items, the first 256 of them one digit each.
constexpr int kPassThreads = 512;
constexpr int kPassWarps = kPassThreads / 32;
constexpr int kIPT = kSortTile / kPassThreads;
constexpr int kLookbackWords = 8;  // predecessors a look-back thread reads per step

// Look-back word: [epoch:30][flag:2][value:32].
constexpr uint64_t kFlagAgg = 1, kFlagIncl = 2;
__device__ __forceinline__ uint64_t lb_pack(uint32_t epoch, uint64_t flag, uint32_t v) {
  return (uint64_t(epoch) << 34) | (flag << 32) | v;
}

struct Loader {
  int mode;
  const uint32_t* keys;
  const uint32_t* vals;
  const uint8_t* del;
  uint32_t n_in;  // ops in the input, 1 .. n
  uint32_t n;

  // Calls f with the mode as a compile-time constant: a loop over elements
  // inside f has no branch on it, so that all its loads are issued before the
  // first is waited for.
  template <class F>
  __device__ __forceinline__ void with_mode(const F& f) const {
    switch (mode) {
      case kSortPairs: return f(Mode<kSortPairs>{});
      case kSortInsert: return f(Mode<kSortInsert>{});
      case kSortDelete: return f(Mode<kSortDelete>{});
      case kSortUpdate: return f(Mode<kSortUpdate>{});
      default: return f(Mode<kSortQueries>{});
    }
  }
  template <int M>
  struct Mode {
    static constexpr int value = M;
    static constexpr bool batch = M != kSortPairs && M != kSortQueries;
  };

  // Where element p of the logical sequence comes from.  Batch modes:
  // position p of the reversed padded batch, i.e. op min(n - 1 - p, n_in - 1).
  template <int M>
  __device__ __forceinline__ uint32_t src(uint32_t p) const {
    return Mode<M>::batch ? min(n - 1 - p, n_in - 1) : p;
  }
  // Delete flag of input s (as loaded: any value but 0 deletes).
  template <int M>
  __device__ __forceinline__ uint32_t flag(uint32_t s) const {
    return M == kSortUpdate ? uint32_t(__ldg(del + s)) : uint32_t(M == kSortDelete);
  }
  // Key variable of an input key with its flag; bad: a key above the user
  // range, which becomes a placebo tombstone.
  template <int M>
  static __device__ __forceinline__ uint32_t encode(uint32_t k, uint32_t fl, bool& bad) {
    if (!Mode<M>::batch) return k;
    const bool b = k > kMaxUserKey;
    bad |= b;
    return b ? kPlaceboKv : ((k << 1) | (fl ? 0u : 1u));
  }
  // Value of element p, as loaded; tombstones (and so bad keys) carry 0.
  template <int M>
  __device__ __forceinline__ uint32_t raw_val(uint32_t p) const {
    return M == kSortQueries ? p : (M == kSortDelete ? 0u : __ldg(vals + src<M>(p)));
  }
  template <int M>
  static __device__ __forceinline__ uint32_t val_of(uint32_t kv, uint32_t raw) {
    return Mode<M>::batch && !(kv & 1u) ? 0u : raw;
  }

  // Leading positions of the reversed padded batch that are padding (copies
  // of op n_in - 1); 0 outside the batch modes.
  __device__ __forceinline__ uint32_t npad() const {
    if (mode == kSortPairs || mode == kSortQueries) return 0u;
    return n - n_in;
  }

  // One element.
  __device__ __forceinline__ void load(uint32_t p, uint32_t& kv, uint32_t& v, bool& bad) const {
    bad = false;
    with_mode([&](auto m) {
      constexpr int M = decltype(m)::value;
      kv = encode<M>(__ldg(keys + src<M>(p)), flag<M>(src<M>(p)), bad);
      v = val_of<M>(kv, raw_val<M>(p));
    });
  }
  __device__ __forceinline__ uint32_t load_key(uint32_t p, bool& bad) const {
    uint32_t kv = 0;
    bad = false;
    with_mode([&](auto m) {
      constexpr int M = decltype(m)::value;
      kv = encode<M>(__ldg(keys + src<M>(p)), flag<M>(src<M>(p)), bad);
    });
    return kv;
  }

  // Elements p0 + step j of a thread, j < N, that pass `in(p)`: all loads
  // first.  Elements outside keep kv = `none` and v = 0.
  template <int N, class In>
  __device__ __forceinline__ void load_keys(uint32_t p0, uint32_t step, const In& in, uint32_t none, uint32_t (&kv)[N],
                                            bool& bad) const {
    with_mode([&](auto m) {
      constexpr int M = decltype(m)::value;
      uint32_t fl[N];
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const uint32_t p = p0 + j * step;
        if (in(p)) {
          kv[j] = __ldg(keys + src<M>(p));
          fl[j] = flag<M>(src<M>(p));
        }
      }
#pragma unroll
      for (int j = 0; j < N; ++j) kv[j] = in(p0 + j * step) ? encode<M>(kv[j], fl[j], bad) : none;
    });
  }
  template <int N, class In>
  __device__ __forceinline__ void load_vals(uint32_t p0, uint32_t step, const In& in, const uint32_t (&kv)[N],
                                            uint32_t (&v)[N]) const {
    with_mode([&](auto m) {
      constexpr int M = decltype(m)::value;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const uint32_t p = p0 + j * step;
        const uint32_t x = kv[j];
        v[j] = in(p) ? raw_val<M>(p) : 0u;
        v[j] = val_of<M>(x, v[j]);
      }
    });
  }
  template <int N, class In>
  __device__ __forceinline__ void load_items(uint32_t p0, uint32_t step, const In& in, uint32_t (&kv)[N],
                                             uint32_t (&v)[N], bool& bad) const {
    uint32_t none;
    load_items<false>(p0, step, in, kv, v, bad, 0u, none);
  }
  // The same, and the key variable of element `at`, asked for behind them.
  template <bool kProbe, int N, class In>
  __device__ __forceinline__ void load_items(uint32_t p0, uint32_t step, const In& in, uint32_t (&kv)[N],
                                             uint32_t (&v)[N], bool& bad, uint32_t at, uint32_t& probe) const {
    with_mode([&](auto m) {
      constexpr int M = decltype(m)::value;
      uint32_t fl[N], probe_fl = 0u;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const uint32_t p = p0 + j * step;
        kv[j] = v[j] = fl[j] = 0u;
        if (in(p)) {
          kv[j] = __ldg(keys + src<M>(p));
          fl[j] = flag<M>(src<M>(p));
          v[j] = raw_val<M>(p);
        }
      }
      if (kProbe) {
        probe = __ldg(keys + src<M>(at));
        probe_fl = flag<M>(src<M>(at));
      }
      bool b = false;  // (of another thread's element)
      if (kProbe) probe = encode<M>(probe, probe_fl, b);
#pragma unroll
      for (int j = 0; j < N; ++j) {
        if (!in(p0 + j * step)) continue;
        kv[j] = encode<M>(kv[j], fl[j], bad);
        v[j] = val_of<M>(kv[j], v[j]);
      }
    });
  }
};

// End of the key check of a sort's first kernel: called by one thread of every
// CTA with whether the CTA saw a key out of range.  The verdict goes to the
// control block; with `host`, the last CTA to get here stores it there too.
struct KeyCheck {
  uint32_t* host;   // null: a deferred check, or none
  uint32_t seq;
  bool on;
  __device__ __forceinline__ void done(uint32_t* ctl, bool bad) const {
    if (!on) return;
    if (bad) {
      atomicOr(ctl + kSortCtlStatus, kErrBadKey);
      __threadfence();
    }
    if (!host || atomicAdd(ctl + kSortCtlChecked, 1u) != gridDim.x - 1) return;
    __threadfence();
    const uint32_t any = atomicOr(ctl + kSortCtlStatus, 0u);
    *reinterpret_cast<volatile uint32_t*>(host) = check_word(seq, any != 0u);
  }
};

// 8 elements a thread at a time, so that as many loads are in flight.
constexpr uint32_t kHistItems = 8, kHistChunk = kHistItems * kPassThreads;
__global__ void __launch_bounds__(kPassThreads) sort_histogram(Loader ld, uint32_t* ctl, KeyCheck check) {
  __shared__ uint32_t s_h[kSortPasses * kRadix];
  for (int i = threadIdx.x; i < kSortPasses * kRadix; i += kPassThreads) s_h[i] = 0;
  __syncthreads();
  bool bad_any = false;
  for (uint64_t p0 = uint64_t(blockIdx.x) * kHistChunk; p0 < ld.n; p0 += uint64_t(gridDim.x) * kHistChunk) {
    uint32_t kv[kHistItems];
    const uint32_t left = uint32_t(ld.n - p0 < kHistChunk ? ld.n - p0 : kHistChunk);
    ld.load_keys(uint32_t(p0) + threadIdx.x, uint32_t(kPassThreads),
                 [&](uint32_t p) { return p - uint32_t(p0) < left; }, 0u, kv, bad_any);
#pragma unroll
    for (uint32_t j = 0; j < kHistItems; ++j) {
      if (j * kPassThreads + threadIdx.x < left) {
#pragma unroll
        for (int d = 0; d < kSortPasses; ++d) atomicAdd(&s_h[d * kRadix + ((kv[j] >> (8 * d)) & 255u)], 1u);
      }
    }
  }
  const int any_bad = __syncthreads_or(bad_any);
  for (int i = threadIdx.x; i < kSortPasses * kRadix; i += kPassThreads) {
    const uint32_t c = s_h[i];
    if (c) atomicAdd(ctl + i, c);
  }
  if (threadIdx.x == 0) check.done(ctl, any_bad != 0);
}

// One 8-bit pass over a tile of 8192 elements, bound by the chain of phases
// of a tile (loads, ranks, look-back, scatter) with two tiles an SM in flight:
// 290 us a pass at n = 5 10^7 (2.8 TB/s of reads and writes).  Tiles of 4096
// in CTAs of 143 registers, one an SM, took 1161 us a pass: the look-back
// advances by at most its window (8 tiles) per round trip to L2, and one CTA an
// SM hides nothing.  Keys are ranked and put in shared memory before the values
// are loaded, so that 16 items a thread fit 64 registers.  Measured beside it
// (the whole sort of 5 10^7 pairs, four passes and the histogram: 1170 us):
// tiles of 6144 at three CTAs an SM 1413 us, of 10240 1258 us, windows of 4 and
// 12 tiles 1207 and 1242 us.
struct PassShared {
  union {
    struct {
      uint32_t keys[kSortTile], vals[kSortTile];
    };
    uint32_t match[kPassWarps][kRadix];  // while ranking: the lanes of the warp that hold the digit
  };
  uint32_t whist[kPassWarps][kRadix];
  uint32_t gbase[kRadix];           // global position of a digit's element minus its tile position
  uint32_t scan[kPassWarps];
  uint32_t tile;
};
constexpr size_t kPassSmem = sizeof(PassShared);

template <bool kFirst>
__global__ void __launch_bounds__(kPassThreads, 2) sort_pass(Loader ld, const uint32_t* __restrict__ in_k,
                                                      const uint32_t* __restrict__ in_v,
                                                      uint32_t* __restrict__ out_k,
                                                      uint32_t* __restrict__ out_v,
                                                      uint32_t* __restrict__ ctl, uint64_t* lookback,
                                                      int pass, uint32_t epoch, uint32_t* sticky) {
  extern __shared__ __align__(16) unsigned char pass_smem[];
  PassShared& sh = *reinterpret_cast<PassShared*>(pass_smem);
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t n = ld.n;
  const int shift = 8 * pass;
  if (tid == 0) sh.tile = atomicAdd(ctl + kSortPasses * kRadix + pass, 1u);
  for (uint32_t i = lane; i < kRadix; i += 32) sh.whist[warp][i] = sh.match[warp][i] = 0;
  __syncthreads();
  const uint32_t tile = sh.tile;
  const uint32_t tile_start = tile * uint32_t(kSortTile);
  const uint32_t tile_n = (n - tile_start) < uint32_t(kSortTile) ? (n - tile_start) : uint32_t(kSortTile);
  const uint32_t e0 = warp * (32 * kIPT) + lane;  // item j: element e0 + 32 j of the tile

  // past the end: the last digit, after every element of it
  uint32_t kv[kIPT], at[kIPT];
  const auto inside = [&](uint32_t p) { return p - tile_start < tile_n; };
  if (kFirst) {
    bool bad = false;
    ld.load_keys(tile_start + e0, 32u, inside, 0xFFFFFFFFu, kv, bad);
  } else {
#pragma unroll
    for (int j = 0; j < kIPT; ++j)
      kv[j] = inside(tile_start + e0 + j * 32) ? __ldg(in_k + tile_start + e0 + j * 32) : 0xFFFFFFFFu;
  }
  const uint32_t hist = tid < kRadix ? ctl[pass * kRadix + tid] : 0u;

  // Rank within the warp, items in (j, lane) order = input order.  The lanes
  // with an item's digit are found by ballots for every other item and
  // through shared memory for the rest: ballots alone kept the ALUs 66 % busy
  // and the shared-memory pipe 44 %, atomics alone 24 % and 55 %.  (All three on
  // the build before the look-back had a thread per digit, whole sorts of 5 10^7
  // pairs: ballots 1368 us, atomics 1466, halves of each 1311; since then 1170.)
  const uint32_t lt = lanemask_lt();
#pragma unroll
  for (int j = 0; j < kIPT; ++j) {
    const uint32_t d = (kv[j] >> shift) & 255u;
    uint32_t peers;
    if (j & 1) {
      atomicOr(&sh.match[warp][d], 1u << lane);
      __syncwarp();
      peers = sh.match[warp][d];
    } else {
      peers = warp_peers<8>(d);
    }
    const uint32_t cnt = sh.whist[warp][d];
    const uint32_t before = __popc(peers & lt);
    __syncwarp();
    if (before == 0) {
      sh.whist[warp][d] = cnt + __popc(peers);
      if (j & 1) sh.match[warp][d] = 0u;
    }
    __syncwarp();
    at[j] = cnt + before;
  }
  __syncthreads();

  // Per digit: warp prefix inside the tile and the tile total (the padding of
  // the last tile taken off the last digit); the tile-local and the global
  // start of the digit.
  uint32_t total = 0;
  if (tid < kRadix) {
#pragma unroll
    for (int w = 0; w < kPassWarps; ++w) total += sh.whist[w][tid];
    if (tid == kRadix - 1) total -= uint32_t(kSortTile) - tile_n;
    // the tile's count is public as early as possible
    st_relaxed_u64(lookback + uint64_t(tile) * kRadix + tid, lb_pack(epoch, tile == 0 ? kFlagIncl : kFlagAgg, total));
  }
  uint32_t sum;
  const uint32_t excl = block_excl_scan<kPassThreads>(total, sh.scan, sum);
  const uint32_t hbase = block_excl_scan<kPassThreads>(hist, sh.scan, sum);
  if (tid < kRadix) {
    uint32_t run = excl;  // each warp's start in the tile
#pragma unroll
    for (int w = 0; w < kPassWarps; ++w) {
      const uint32_t c = sh.whist[w][tid];
      sh.whist[w][tid] = run;
      run += c;
    }
  }
  __syncthreads();

  // Into shared memory in digit order (stable), values last.
#pragma unroll
  for (int j = 0; j < kIPT; ++j) {
    const uint32_t d = (kv[j] >> shift) & 255u;
    at[j] += sh.whist[warp][d];
    sh.keys[at[j]] = kv[j];
  }
  if (kFirst) {
    ld.load_vals(tile_start + e0, 32u, inside, kv, kv);
  } else {
#pragma unroll
    for (int j = 0; j < kIPT; ++j)
      if (inside(tile_start + e0 + j * 32)) kv[j] = __ldg(in_v + tile_start + e0 + j * 32);
  }
#pragma unroll
  for (int j = 0; j < kIPT; ++j) sh.vals[at[j]] = kv[j];

  // Decoupled look-back, one thread per digit, kLookbackWords predecessors
  // per step: the words are consumed from the nearest tile down until an
  // inclusive prefix is found; a word not yet published ends the step, which
  // is then retried from there (bounded in time).
  if (tid < kRadix) {
    uint32_t prefix = 0;
    if (tile) {
      const uint32_t tag_agg = (epoch << 2) | uint32_t(kFlagAgg), tag_incl = (epoch << 2) | uint32_t(kFlagIncl);
      int64_t t = int64_t(tile) - 1;  // nearest predecessor not yet consumed
      uint64_t t0 = 0;
      for (bool incl = false; !incl;) {
        uint64_t w[kLookbackWords];
#pragma unroll
        for (int i = 0; i < kLookbackWords; ++i)
          w[i] = t - i >= 0 ? ld_relaxed_u64(lookback + uint64_t(t - i) * kRadix + tid)
                            : lb_pack(epoch, kFlagIncl, 0u);
        int consumed = 0;
        bool stall = false;
#pragma unroll
        for (int i = 0; i < kLookbackWords; ++i) {
          const uint32_t tag = uint32_t(w[i] >> 32);
          if (!incl && !stall) {
            incl = tag == tag_incl;
            stall = !incl && tag != tag_agg;
            if (!stall) {
              prefix += uint32_t(w[i]);
              ++consumed;
            }
          }
        }
        t -= consumed;
        if (!incl && consumed == 0 && !spin_continue(t0, kWaitLimitNs, sticky)) break;
        if (consumed) t0 = 0;
      }
      st_relaxed_u64(lookback + uint64_t(tile) * kRadix + tid, lb_pack(epoch, kFlagIncl, prefix + total));
    }
    sh.gbase[tid] = hbase - excl + prefix;
  }
  __syncthreads();

  for (uint32_t i = tid; i < tile_n; i += kPassThreads) {
    const uint32_t k = sh.keys[i];
    const uint32_t dst = sh.gbase[(k >> shift) & 255u] + i;
    if (dst < n) {
      out_k[dst] = k;
      out_v[dst] = sh.vals[i];
    }
  }
}

// ---------------------------------------------------------------------------
// Bucket sort for n <= kMsdMaxN (the batch sizes of the plain form): 256 key
// ranges ("buckets") first, then the elements of each.  Two kernels, so that
// a batch sort is one dependent launch after another:
//   msd_tile     per 4096-element tile of the (encoded, reversed) input: the
//                tile stably sorted by bucket in shared memory and written
//                back to the scratch at the tile's own place (one coalesced
//                write), so bucket d's elements of tile t form the run
//                runs[d][t] = (start, count) there; the grand total of each
//                bucket (global atomics) and the key check.
//   bucket_sort  per bucket, one CTA: the bucket's runs, in tile order (the
//                stable order), gathered into shared memory -- the start of
//                the bucket in the output is the sum of the totals before
//                it, so no tile waits for another -- then sorted and written
//                out with the prefix index entries of the bins that start in
//                its range.  A bucket above kBucketCap elements (many copies
//                of a few keys, or keys in clusters) is taken by the same
//                CTA in parts that fit or in 8-bit passes (sort_big).
// The buckets split the range of the keys that the batch holds (KeyMap), not
// the 32 bits of the key variable: ids below 2^25 would otherwise fall in
// four buckets and be sorted by four CTAs; hot keys have buckets of their own.
// ---------------------------------------------------------------------------
constexpr int kBucketThreads = 512;
constexpr int kBucketWarps = kBucketThreads / 32;
constexpr int kBucketIPT = 10;
constexpr uint32_t kBucketCap = kBucketThreads * kBucketIPT;  // 5120
constexpr uint32_t kSubBinMax = 48;      // larger sub-bins take the pass-by-pass path

// The tile kernel runs 512 threads of 8 elements per 4096-element tile:
// many warps to keep loads in flight, and a short ranking chain per warp.
constexpr int kScatterThreads = 512;
constexpr int kScatterWarps = kScatterThreads / 32;
constexpr int kScatterIPT = int(kMsdTile) / kScatterThreads;  // 8
static_assert(kScatterIPT * kScatterThreads == int(kMsdTile), "tile");
static_assert(kMsdMaxTiles <= uint32_t(kBucketThreads), "one thread per tile run in the bucket kernel");

// The buckets of one sort (KeyMap): 256 in all.  lo, mul and the hot ones come
// from 512 elements taken at even distances (every CTA of the tile kernel reads
// the same ones): the range is the one they span, widened at both ends (elements
// beyond it fall in the first or last bucket); hot is what comes up kHotSamples
// times or more, about 0.8 % of the batch, and would overflow a bucket of
// 2^20 / 256 elements.
// With the top byte as the bucket, batches of 2^18 ids below 2^25 took 553 us
// in bucket_sort and 2^20 keys below 2^30 154 us; now 21.7 and 21.3 us.  Without
// buckets for the hot keys a sort of 2^18 Zipf(1.1) pairs took 63 us, of 2^20
// 167; now 34 and 79.
constexpr uint32_t kHotSamples = 4, kMaxHot = 32, kSamples = 512;
constexpr uint32_t kMaxSampledHot = kSamples / kHotSamples;
constexpr int kSampleTableLog = 10, kSampleCellsLog = 12;
constexpr uint32_t kSampleTable = 1u << kSampleTableLog, kSampleCells = 1u << kSampleCellsLog;
// Stores the smallest key variable of every bucket (threads 0 .. 255).
__device__ __forceinline__ void store_bounds(const KeyMap& map, uint32_t* out) {
  const uint32_t t = threadIdx.x;
  if (t < map.parts) {
    const uint32_t kv = t ? map.lower(t) : 0u;
    uint32_t d = t;
    for (uint32_t h = 0; h < map.nhot; ++h) d += map.hot[h] < kv ? 2u : 0u;
    out[d] = kv;
  }
  if (t < map.nhot) {
    const uint32_t d = map.part(map.hot[t]) + 2u * t;
    out[d + 1] = map.hot[t];
    out[d + 2] = map.hot[t] + 1u;
  }
}
static_assert(kRadix == 256 && 2 * kMaxHot < kRadix, "the hot keys' buckets leave parts over");
static_assert(kSamples == uint32_t(kScatterThreads), "one sample a thread");
static_assert(kSampleTable == 2 * kSamples && 2 * kSampleTable == 4 * uint32_t(kScatterThreads) &&
                  2 * kSampleTable <= kSampleCells && kSampleCells <= uint32_t(kMsdTile), "room to count in");

struct SampleShared {
  uint32_t mn[kScatterWarps], mx[kScatterWarps], hot[kMaxHot], n_hot;
};
// Key map of the batch of cnt elements (every thread of the CTA gets it); kv:
// the thread's sample.  First the samples are counted by a hash of theirs: for
// most batches no cell fills up (with 4096 cells a batch of different keys
// fills one in 30 times; 1024 would be filled nearly every time, for 1.3 us).
// Otherwise those in a full cell are counted by key variable, in an open hash
// table half full at most (keys in `cells`, 0 where empty, counts behind
// them).  cells: kSampleCells words of shared memory, 16-byte aligned; list:
// kMaxSampledHot words.  sample_begin comes first, with a barrier between.
__device__ __forceinline__ void sample_begin(const uint32_t kv, uint32_t* cells, SampleShared& sh) {
  const uint32_t tid = threadIdx.x, warp = tid >> 5;
  for (uint32_t i = tid; i < kSampleCells / 4; i += kScatterThreads)
    reinterpret_cast<uint4*>(cells)[i] = make_uint4(0u, 0u, 0u, 0u);
  const uint32_t mn = __reduce_min_sync(0xffffffffu, kv), mx = __reduce_max_sync(0xffffffffu, kv);
  if (lane_id() == 0) {
    sh.mn[warp] = mn;
    sh.mx[warp] = mx;
  }
  if (tid == 0) sh.n_hot = 0u;
}
__device__ __forceinline__ KeyMap sample_map(const uint32_t kv, uint32_t cnt, uint32_t* cells, uint32_t* list,
                                             SampleShared& sh) {
  const uint32_t tid = threadIdx.x;
  const bool seek_hot = cnt >= 8 * kSamples;  // (else elements are sampled twice)
  const uint32_t w = lane_id() & uint32_t(kScatterWarps - 1);
  const uint32_t lo = __reduce_min_sync(0xffffffffu, sh.mn[w]), hi = __reduce_max_sync(0xffffffffu, sh.mx[w]);
  uint32_t nhot = 0;
  if (seek_hot) {
    const uint32_t hash = kv * 0x9E3779B1u, cell = hash >> (32 - kSampleCellsLog);
    atomicAdd(&cells[cell], 1u);
    __syncthreads();
    // (0 has nothing below it, 2^32 - 1 nothing above)
    const bool may = cells[cell] >= kHotSamples && kv != 0u && kv != 0xFFFFFFFFu;
    if (__syncthreads_or(may)) {
      uint32_t *table = cells, *count = cells + kSampleTable, at = hash >> (32 - kSampleTableLog);
      reinterpret_cast<uint4*>(cells)[tid] = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();
      bool first = false;  // the sample that entered its key variable
      if (may) {
        for (;;) {
          uint32_t was = reinterpret_cast<volatile uint32_t*>(table)[at];
          if (was == 0u) {
            was = atomicCAS(&table[at], 0u, kv);
            first = was == 0u;
          }
          if (first || was == kv) break;
          at = (at + 1u) & (kSampleTable - 1u);
        }
        atomicAdd(&count[at], 1u);
      }
      __syncthreads();
      if (first && count[at] >= kHotSamples) list[atomicAdd(&sh.n_hot, 1u)] = kv;
      __syncthreads();
      // at most kMaxSampledHot of them, of which the kMaxHot lowest are taken, in order
      nhot = sh.n_hot;
      if (tid < nhot) {
        const uint32_t x = list[tid];
        uint32_t r = 0;
        for (uint32_t i = 0; i < nhot; ++i) r += list[i] < x ? 1u : 0u;
        if (r < kMaxHot) sh.hot[r] = x;
      }
      nhot = min(nhot, kMaxHot);
      __syncthreads();
    }
  }
  return KeyMap::spanning(lo, hi, uint32_t(kRadix) - 2u * nhot, nhot, sh.hot);
}

// Stable in-shared-memory rank of up to IPT items per thread of a warp-striped
// block (item j of lane l of warp w is element w*32*IPT + j*32 + l): on return
// s_whist[w][d] holds warp w's start inside digit d's run, s_excl[d] the run's
// start, and rank[j] the item's position among its warp's items of its digit.
// digit(kv) is below kRadix.  With ipt < IPT only the first ipt items of each
// thread are ranked (the caller lays the block out with 32 ipt items a warp).
template <int NT, int IPT, class Digit>
__device__ __forceinline__ void rank_block(const uint32_t (&kv)[IPT], uint32_t m, uint32_t base, const Digit& digit,
                                           uint32_t (&rank)[IPT], uint32_t (*s_whist)[kRadix],
                                           uint32_t* s_excl, uint32_t* s_scan, uint32_t* digit_total,
                                           uint32_t lo = 0, int ipt = IPT) {
  constexpr int NW = NT / 32;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  for (uint32_t i = lane; i < kRadix; i += 32) s_whist[warp][i] = 0;
  __syncwarp();
  const uint32_t lt = lanemask_lt();
#pragma unroll
  for (int j = 0; j < IPT; ++j) {
    if (j >= ipt) break;  // the same for the whole block
    const uint32_t p = base + j * 32 + lane;
    const uint32_t d = (p < m && p >= lo) ? digit(kv[j]) : kNoDigit;
    const uint32_t peers = warp_peers<9>(d);  // d <= kNoDigit = 256
    const uint32_t before = __popc(peers & lt);
    const uint32_t cnt = (d != kNoDigit) ? s_whist[warp][d] : 0u;
    __syncwarp();
    if (d != kNoDigit && before == 0) s_whist[warp][d] = cnt + __popc(peers);
    __syncwarp();
    rank[j] = cnt + before;
  }
  __syncthreads();
  uint32_t total = 0;
  if (tid < kRadix) {
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const uint32_t c = s_whist[w][tid];
      s_whist[w][tid] = total;
      total += c;
    }
  }
  uint32_t all;
  const uint32_t excl = block_excl_scan<NT>(tid < kRadix ? total : 0u, s_scan, all);
  if (tid < kRadix) {
    s_excl[tid] = excl;
    if (digit_total) digit_total[tid] = total;
  }
  __syncthreads();
}

// The padding of a short batch (copies of its last op, the leading
// positions of the reversed sequence) is neither ranked nor written: it is
// one run of equal elements, added to its bucket's total here and written by
// that bucket's sort at its sorted place.  A tile of padding only still
// writes its (empty) runs.
// 48 registers (a few spills): with the 62 that the compiler would take, fewer
// CTAs find room beside those of the fold before them, and 128 inserts of
// 2^20 took 1 to 2 % longer.
__global__ void __maxnreg__(48) msd_tile(Loader ld, uint32_t* __restrict__ tmp_k,
                                                     uint32_t* __restrict__ tmp_v, uint2* __restrict__ runs,
                                                     uint32_t* ctl, KeyCheck check) {
  __shared__ __align__(16) uint32_t s_keys[kMsdTile];
  __shared__ __align__(16) uint32_t s_vals[kMsdTile];
  __shared__ uint32_t s_whist[kScatterWarps][kRadix];
  __shared__ uint32_t s_excl[kRadix], s_cnt[kRadix], s_scan[kScatterWarps];
  __shared__ SampleShared s_sample;
  pdl_trigger();
  pdl_wait();
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, tile = blockIdx.x;
  const uint32_t n = ld.n, npad = ld.npad();
  const uint32_t t0 = tile * kMsdTile;
  const uint32_t base = t0 + warp * (32 * kScatterIPT);
  uint32_t kv[kScatterIPT], v[kScatterIPT];
  bool bad_any = false;
  uint32_t sample;
  ld.load_items<true>(base + lane, 32u, [&](uint32_t p) { return p < n && p >= npad; }, kv, v, bad_any,
                      npad + uint32_t(uint64_t(tid) * (n - npad) / kSamples), sample);
  sample_begin(sample, s_keys, s_sample);
  const int any_bad = __syncthreads_or(bad_any);
  if (tid == 0) check.done(ctl, any_bad != 0);
  const KeyMap map = sample_map(sample, n - npad, s_keys, s_vals, s_sample);
  if (tile == gridDim.x - 1) {  // the last tile's CTA (the shortest) publishes the buckets' bounds
    store_bounds(map, ctl + kSortCtlBounds);
    if (tid == kRadix) {
      ctl[kSortCtlMap] = map.lo;
      ctl[kSortCtlMap + 1] = map.mul;
    }
  }
  // ranked and put in order in shared memory; digit(x[j]) is element j's bucket
  const auto place = [&](const uint32_t (&x)[kScatterIPT], const auto& digit) {
    uint32_t rank[kScatterIPT];
    rank_block<kScatterThreads, kScatterIPT>(x, n, base, digit, rank, s_whist, s_excl, s_scan, s_cnt, npad);
#pragma unroll
    for (int j = 0; j < kScatterIPT; ++j) {
      const uint32_t p = base + j * 32 + lane;
      if (p < n && p >= npad) {
        const uint32_t d = digit(x[j]);
        const uint32_t pos = s_excl[d] + s_whist[warp][d] + rank[j];
        s_keys[pos] = kv[j];
        s_vals[pos] = v[j];
      }
    }
  };
  if (map.nhot == 0) {
    place(kv, [&](uint32_t k) { return map.part(k); });
  } else {
    uint32_t dig[kScatterIPT];
#pragma unroll
    for (int j = 0; j < kScatterIPT; ++j) dig[j] = map.part(kv[j]);
#pragma unroll 1
    for (uint32_t h = 0; h < map.nhot; ++h) {
      const uint32_t x = map.hot[h];
#pragma unroll
      for (int j = 0; j < kScatterIPT; ++j) dig[j] += (kv[j] >= x ? 1u : 0u) + (kv[j] > x ? 1u : 0u);
    }
    place(dig, [](uint32_t d) { return d; });
  }
  __syncthreads();
  const uint32_t lo_t = t0 > npad ? t0 : npad, hi_t = (n - t0) < kMsdTile ? n : t0 + kMsdTile;
  const uint32_t tile_n = hi_t > lo_t ? hi_t - lo_t : 0u;  // real elements of the tile
  for (uint32_t i = tid; i < tile_n; i += kScatterThreads) {
    tmp_k[t0 + i] = s_keys[i];
    tmp_v[t0 + i] = s_vals[i];
  }
  if (tid < kRadix) {
    const uint32_t c = s_cnt[tid];
    runs[tid * kMsdMaxTiles + tile] = make_uint2(t0 + s_excl[tid], c);
    if (c) atomicAdd(ctl + 3 * kRadix + tid, c);
  }
  if (tile == 0 && tid == 0 && npad) {
    bool bad;
    atomicAdd(ctl + 3 * kRadix + map.bucket(ld.load_key(0, bad)), npad);
  }
}

// First position i in [0, m) with a[i] >= kv, a sorted.
__device__ __forceinline__ uint32_t lower_bound_sorted(const uint32_t* a, uint32_t m, uint32_t kv) {
  uint32_t lo = 0, hi = m;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (a[mid] < kv) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// A bucket: its elements' key variables lie in [lo, hi]; `map` spreads them
// over the sub-bins of the counting pass.
struct BucketRange {
  uint32_t lo, hi;
  SubMap map;
};
struct PadRun {   // n copies of (kv, v) that belong to the bucket but are not among its elements
  uint32_t n, kv, v;
};
struct BinRange {  // prefix-index entries [bin0, bin1) to write (bin P starts at key variable P << fshift)
  uint32_t* fence;
  int fshift;
  uint32_t bin0, bin1;
};

// A bucket after its sort, for reading back: either sorted (cnt null), or in
// sub-bins in no order, cnt[s] being the first position of sub-bin s.
struct SortedView {
  const uint32_t* a;
  uint32_t m;
  const uint32_t* cnt;
  SubMap map;
  __device__ __forceinline__ uint32_t end(uint32_t s) const { return s + 1 < kSubBins ? cnt[s + 1] : m; }
  // number of elements below kv
  __device__ __forceinline__ uint32_t less(uint32_t kv) const {
    if (!cnt) return lower_bound_sorted(a, m, kv);
    const uint32_t s = map.sub(kv), e = end(s);
    uint32_t c = cnt[s];
    for (uint32_t y = c; y < e; ++y) c += a[y] < kv ? 1u : 0u;
    return c;
  }
  __device__ __forceinline__ uint32_t smallest() const {
    uint32_t k = a[0];
    if (cnt)
      for (uint32_t y = 1, e = end(map.sub(k)); y < e; ++y) k = min(k, a[y]);
    return k;
  }
  __device__ __forceinline__ uint32_t largest() const {
    uint32_t k = a[m - 1];
    if (cnt)
      for (uint32_t y = cnt[map.sub(k)]; y < m; ++y) k = max(k, a[y]);
    return k;
  }
};

// Where element i of a bucket lives in the scratch its sort reads.
// ContigSrc: elements start .. start + m - 1 (the batched form's scatter
// writes every bucket contiguously).  RunSrc: the bucket's runs over the
// tiles, in tile order (the stable order); rstart[t] is the first bucket
// position of run t (an exclusive scan of the run lengths) and run t's
// element i - rstart[t] sits at rbase[t] + i (both in shared memory).
// at(i) serves buckets in shared memory; find(i) any; seek(i, t) any, for i
// that never go down from call to call (t starts at 0 and follows the runs).
struct ContigSrc {
  uint32_t start;
  __device__ __forceinline__ uint32_t at(uint32_t i) const { return start + i; }
  __device__ __forceinline__ uint32_t find(uint32_t i) const { return start + i; }
  __device__ __forceinline__ uint32_t seek(uint32_t i, uint32_t&) const { return start + i; }
};
struct RunSrc {
  const uint32_t* rstart;  // nruns + 1 entries, rstart[nruns] = the bucket's size
  const uint32_t* rbase;
  const uint8_t* chunk;    // run holding element 16 c, per 16-element chunk c (buckets in shared memory only)
  uint32_t nruns;          // >= 1
  __device__ __forceinline__ uint32_t at(uint32_t i) const {
    uint32_t t = chunk[i >> 4];  // from the run of the chunk's first element, forward (runs of ~16 elements)
    return seek(i, t);
  }
  // the run holding i: the largest t with rstart[t] <= i (empty runs share
  // their start with the next run, so they are never the largest)
  __device__ __forceinline__ uint32_t seek(uint32_t i, uint32_t& t) const {
    while (rstart[t + 1] <= i) ++t;
    return rbase[t] + i;
  }
  __device__ __forceinline__ uint32_t find(uint32_t i) const {
    uint32_t lo = 0, hi = nruns - 1;
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (rstart[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return rbase[lo] + i;
  }
};
static_assert(kMsdMaxTiles <= 256u, "a run index fits in a byte");

// Shared memory of a bucket's CTA.
struct BucketShared {
  uint32_t whist[kBucketWarps][kRadix];  // also the kSubBins counters
  uint32_t excl[kRadix], scan[kBucketWarps];
  uint32_t max, cnt[3], mn, mx;
  uint64_t scan64[kBucketWarps];
  uint32_t cand[kBucketWarps], votes[kBucketWarps];
};

// Sorts m <= kBucketCap elements stably by the key variable (all in
// [range.lo, range.hi]) and hands each to emit(position, kv, value).
// load(kv, v) fills a thread's elements threadIdx.x + j kBucketThreads (< m) of
// the stable order; with kHeld they come from bsm, which holds all of them in
// order (kBucketCap words of keys, then the values).
//   Fast path (no sub-bin above kSubBinMax): one counting pass places every
//   element in its sub-bin (about one element each for spread keys), at an
//   arbitrary slot; every element is then emitted at its sub-bin's start plus
//   its rank in the sub-bin by (key variable, index), the stable order.  Its
//   place differs from its slot by less than a sub-bin, so the caller's
//   stores are nearly in order.
//   Otherwise stable 8-bit passes over the bits in which the range differs.
// bsm holds 4 kBucketCap words plus kBucketCap 16-bit indexes.  The view
// returned stays valid until bsm or sh.whist change.
template <bool kHeld, class Load, class Emit>
__device__ __forceinline__ SortedView sort_resident(const Load& load, uint32_t m, const BucketRange& range,
                                                    uint32_t* bsm, BucketShared& sh, const Emit& emit) {
  static_assert(kSubBins == kBucketWarps * kRadix, "the counters reuse the per-warp histograms");
  uint32_t *ak = bsm, *av = bsm + kBucketCap, *bk = bsm + 2 * kBucketCap, *bv = bsm + 3 * kBucketCap;
  uint16_t* bi = reinterpret_cast<uint16_t*>(bsm + 4 * kBucketCap);
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  uint32_t* cnt = &sh.whist[0][0];
  uint32_t kv[kBucketIPT], v[kBucketIPT];
  load(kv, v);
  for (uint32_t i = tid; i < kSubBins; i += kBucketThreads) cnt[i] = 0u;
  if (tid == 0) sh.max = 0u;
  __syncthreads();
  uint32_t slot[kBucketIPT];  // sub-bin, and above bit 16 the slot there
#pragma unroll
  for (int j = 0; j < kBucketIPT; ++j) {
    if (tid + j * kBucketThreads < m) {
      const uint32_t sb = range.map.sub(kv[j]);
      slot[j] = sb | (atomicAdd(&cnt[sb], 1u) << 16);
    }
  }
  __syncthreads();
  // sub-bin starts: thread t owns counters [8 t, 8 t + 8)
  constexpr int kPer = int(kSubBins) / kBucketThreads;
  uint32_t c[kPer], sum = 0, mx = 0;
#pragma unroll
  for (int e = 0; e < kPer; ++e) {
    c[e] = cnt[tid * kPer + e];
    sum += c[e];
    mx = max(mx, c[e]);
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0 && mx > kSubBinMax) atomicMax(&sh.max, mx);
  uint32_t all;
  uint32_t run = block_excl_scan<kBucketThreads>(sum, sh.scan, all);
  if (sh.max <= kSubBinMax) {  // uniform: sh.max settled before the scan's barriers
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      cnt[tid * kPer + e] = run;
      run += c[e];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kBucketIPT; ++j) {
      const uint32_t i = tid + j * kBucketThreads;
      if (i < m) {
        const uint32_t pos = cnt[slot[j] & 0xFFFFu] + (slot[j] >> 16);
        bk[pos] = kv[j];
        bv[pos] = v[j];
        bi[pos] = uint16_t(i);
      }
    }
    __syncthreads();
    // Each element counts the members of its sub-bin that precede it
    // (independent loads, about two a sub-bin for spread keys) rather than a
    // per-sub-bin insertion sort, whose shifting chain made a warp wait for
    // its fullest sub-bin.
    const SortedView view{bk, m, cnt, range.map};
#pragma unroll 2
    for (int j = 0; j < kBucketIPT; ++j) {
      const uint32_t x = tid + j * kBucketThreads;
      if (x < m) {
        const uint32_t k = bk[x], vv = bv[x];
        const uint32_t b = range.map.sub(k);
        const uint32_t s0 = cnt[b], s1 = view.end(b);
        // The first four members without a branch (a sub-bin rarely holds
        // more for spread keys, and a loop made each warp run as long as
        // its fullest sub-bin), then the rest; equal key variables, which
        // are rare too, are told apart by index afterwards.
        uint32_t r = 0, eq = 0;
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
          const uint32_t ky = s0 + u < s1 ? bk[s0 + u] : 0xFFFFFFFFu;
          r += ky < k ? 1u : 0u;
          eq += ky == k ? 1u : 0u;
        }
        for (uint32_t y = s0 + 4; y < s1; ++y) {
          r += bk[y] < k ? 1u : 0u;
          eq += bk[y] == k ? 1u : 0u;
        }
        if (eq > 1) {
          const uint16_t ix = bi[x];
          for (uint32_t y = s0; y < s1; ++y) r += bk[y] == k && bi[y] < ix ? 1u : 0u;
        }
        emit(s0 + r, k, vv);
      }
    }
    return view;
  }
  __syncthreads();
  // Many copies of one key, or a cluster.  The block is laid out with as many
  // items a thread as m needs, so that a small bucket's passes are short.
  if (!kHeld) {
#pragma unroll
    for (int j = 0; j < kBucketIPT; ++j) {
      const uint32_t i = tid + j * kBucketThreads;
      if (i < m) {
        ak[i] = kv[j];
        av[i] = v[j];
      }
    }
    __syncthreads();
  }
  const int ipt = int((m + kBucketThreads - 1) / kBucketThreads);
  const uint32_t wbase = warp * 32u * uint32_t(ipt);
  const int bits = 32 - __clz(int(range.hi - range.lo));
  uint32_t rank[kBucketIPT];
  for (int shift = 0; shift < bits; shift += 8) {
#pragma unroll
    for (int j = 0; j < kBucketIPT; ++j) {
      if (j >= ipt) break;
      const uint32_t p = wbase + j * 32 + lane;
      kv[j] = p < m ? ak[p] : 0u;
      v[j] = p < m ? av[p] : 0u;
    }
    const auto digit = [&](uint32_t k) { return ((k - range.lo) >> shift) & 255u; };
    rank_block<kBucketThreads, kBucketIPT>(kv, m, wbase, digit, rank, sh.whist, sh.excl, sh.scan, nullptr, 0u, ipt);
#pragma unroll
    for (int j = 0; j < kBucketIPT; ++j) {
      if (j >= ipt) break;
      const uint32_t p = wbase + j * 32 + lane;
      if (p < m) {
        const uint32_t dg = digit(kv[j]);
        const uint32_t pos = sh.excl[dg] + sh.whist[warp][dg] + rank[j];
        bk[pos] = kv[j];
        bv[pos] = v[j];
      }
    }
    __syncthreads();
    uint32_t* t;
    t = ak; ak = bk; bk = t;
    t = av; av = bv; bv = t;
  }
  for (uint32_t i = tid; i < m; i += kBucketThreads) emit(i, ak[i], av[i]);
  return SortedView{ak, m, nullptr, range.map};
}

// A bucket above kBucketCap elements of many different keys in clusters: stable
// 8-bit passes over the bits in which the keys [mn, mx] differ, kBucketCap
// elements at a time, between the bucket's places in the scratch and out[0 .. m)
// (every element is read and written once per pass, whatever the keys; pass 0
// reads the scratch).  The last pass leaves room for the padding run.  Bound by
// the one CTA's instructions, about 9 us a chunk.
template <class Src>
__device__ __noinline__ void sort_digits(uint32_t* src_k, uint32_t* src_v, const Src src, uint32_t* out_k,
                                         uint32_t* out_v, uint32_t m, uint32_t mn, uint32_t mx, const PadRun pad,
                                         uint32_t* bsm, BucketShared& sh) {
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  uint32_t *to = bsm, *tot = to + kSortPasses * kRadix;  // next place of a digit per pass, its count in the chunk
  uint32_t *sk = tot + kRadix, *sv = sk + kBucketCap;
  static_assert((kSortPasses + 1) * kRadix <= kBucketCap, "fits the bucket's shared memory");
  const int passes = (32 - __clz(int(mx - mn)) + 7) / 8;
  const auto room = [&](uint32_t kv) { return pad.n && kv >= pad.kv ? pad.n : 0u; };
  for (uint32_t i = tid; i < uint32_t(kSortPasses * kRadix); i += kBucketThreads) to[i] = 0u;
  __syncthreads();
  constexpr uint32_t kItems = 8;
  for (uint32_t i0 = 0, t = 0; i0 < m; i0 += kItems * kBucketThreads) {
    uint32_t k[kItems];
#pragma unroll
    for (uint32_t j = 0; j < kItems; ++j) {
      const uint32_t i = i0 + j * kBucketThreads + tid;
      k[j] = i < m ? src_k[src.seek(i, t)] - mn : 0u;
    }
#pragma unroll
    for (uint32_t j = 0; j < kItems; ++j)
      if (i0 + j * kBucketThreads + tid < m)
        for (int p = 0; p < passes; ++p) atomicAdd(&to[p * kRadix + ((k[j] >> (8 * p)) & 255u)], 1u);
  }
  __syncthreads();
  for (int p = 0; p < passes; ++p) {
    uint32_t all;
    const uint32_t first = block_excl_scan<kBucketThreads>(tid < kRadix ? to[p * kRadix + tid] : 0u, sh.scan, all);
    if (tid < kRadix) to[p * kRadix + tid] = first;
  }
  __syncthreads();
  const uint32_t wbase = warp * (32 * kBucketIPT);
  for (int p = 0; p < passes; ++p) {
    const bool back = p & 1;  // out -> scratch
    const auto digit = [&](uint32_t k) { return ((k - mn) >> (8 * p)) & 255u; };
    for (uint32_t c0 = 0, t = 0; c0 < m; c0 += kBucketCap) {
      const uint32_t cm = min(m - c0, kBucketCap);
      uint32_t kv[kBucketIPT], v[kBucketIPT], rank[kBucketIPT];
#pragma unroll
      for (int j = 0; j < kBucketIPT; ++j) {
        const uint32_t x = wbase + j * 32 + lane;
        kv[j] = v[j] = 0u;
        if (x < cm) {
          const uint32_t at = back ? c0 + x : src.seek(c0 + x, t);
          kv[j] = back ? out_k[at] : src_k[at];
          v[j] = back ? out_v[at] : src_v[at];
        }
      }
      rank_block<kBucketThreads, kBucketIPT>(kv, cm, wbase, digit, rank, sh.whist, sh.excl, sh.scan, tot);
#pragma unroll
      for (int j = 0; j < kBucketIPT; ++j) {
        if (wbase + j * 32 + lane < cm) {
          const uint32_t d = digit(kv[j]), at = sh.excl[d] + sh.whist[warp][d] + rank[j];
          sk[at] = kv[j];
          sv[at] = v[j];
        }
      }
      __syncthreads();
      for (uint32_t i = tid; i < cm; i += kBucketThreads) {
        const uint32_t k = sk[i], d = digit(k), at = to[p * kRadix + d] + (i - sh.excl[d]);
        if (back) {
          const uint32_t x = src.find(at);
          src_k[x] = k;
          src_v[x] = sv[i];
        } else {
          const uint32_t x = p + 1 == passes ? at + room(k) : at;
          out_k[x] = k;
          out_v[x] = sv[i];
        }
      }
      __syncthreads();
      if (tid < kRadix) to[p * kRadix + tid] += tot[tid];
    }
  }
  if (passes & 1) return;
  uint32_t t = 0;  // an even number of passes ends in the scratch
  for (uint32_t i0 = 0; i0 < m; i0 += kItems * kBucketThreads) {
    uint32_t k[kItems], v[kItems];
#pragma unroll
    for (uint32_t j = 0; j < kItems; ++j) {
      const uint32_t i = i0 + j * kBucketThreads + tid;
      const uint32_t at = i < m ? src.seek(i, t) : 0u;
      k[j] = i < m ? src_k[at] : 0u;
      v[j] = i < m ? src_v[at] : 0u;
    }
#pragma unroll
    for (uint32_t j = 0; j < kItems; ++j) {
      const uint32_t i = i0 + j * kBucketThreads + tid;
      if (i < m) {
        out_k[i + room(k[j])] = k[j];
        out_v[i + room(k[j])] = v[j];
      }
    }
  }
}

// A bucket above kBucketCap elements: taken in key order, a part at a time.
// Each round looks at the elements of [a, b], the keys still to do (KeyTurn):
//   at most kBucketCap of them        gathered in order, sorted, written;
//   all but at most kBucketCap have   the hot key's tombstones and regular
//   one key (a hot key)               elements go straight to their places in
//                                     order, the others as above, around them;
//   otherwise                         b is lowered to the end of the longest
//                                     prefix of sub-bins that fits.
// A round reads the bucket two or three times (from L2), 8 independent loads
// a thread at a time.  Bound by the one CTA's chain of rounds.  (sort_digits
// alone: a sort of 2^20 pairs of which 8 % have one key 448 us, with the rounds
// 164.)  Their time grows with the square of the bucket, so more than kMaxParts *
// kBucketCap elements beside the hot key are left to sort_digits: 2^18 keys, as
// many in every octave, 15.1 -> 1.26 ms, 2^20 178 -> 4.6; 2^20 of which 2 % lie
// anywhere and the rest below 2^24 109 -> 3.0; in ten clusters 5.9 -> 0.66.  At
// three parts 2^14 such keys take 120 us, at two 102; below two the rounds are
// the faster ones (four rounds of 128 batches of 8192 keys whose larger bucket
// holds 5500: 443 us, with the passes 565).
constexpr uint32_t kMaxParts = 2;
template <class Src>
__device__ __noinline__ void sort_big(uint32_t* src_k, uint32_t* src_v, const Src src, uint32_t* out_k,
                                      uint32_t* out_v, uint32_t start, uint32_t m, const BucketRange range,
                                      const PadRun pad, uint32_t* bsm, BucketShared& sh) {
  constexpr uint32_t kItems = 8, kChunk = kItems * kBucketThreads;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  if (range.lo == range.hi) {  // a hot key's bucket: its elements in order, after the padding if that is of the key
    const uint32_t base = start + pad.n;
    for (uint32_t j = tid; j < pad.n; j += kBucketThreads) {
      out_k[start + j] = pad.kv;
      out_v[start + j] = pad.v;
    }
    constexpr uint32_t kFar = 24;  // loads in flight (one CTA copies 3.3 elements a nanosecond)
    uint32_t t = 0;
    for (uint32_t i0 = 0; i0 < m; i0 += kFar * kBucketThreads) {
      uint32_t v[kFar];
#pragma unroll
      for (uint32_t j = 0; j < kFar; ++j) {
        const uint32_t i = i0 + j * kBucketThreads + tid;
        v[j] = i < m ? src_v[src.seek(i, t)] : 0u;
      }
#pragma unroll
      for (uint32_t j = 0; j < kFar; ++j) {
        const uint32_t i = i0 + j * kBucketThreads + tid;
        if (i < m) {
          out_k[base + i] = range.lo;
          out_v[base + i] = v[j];
        }
      }
    }
    __syncthreads();  // the caller reads the output back
    return;
  }
  uint32_t* cnt = &sh.whist[0][0];
  const auto shift = [&](uint32_t kv) { return pad.n && kv >= pad.kv ? pad.n : 0u; };
  // f(kv, valid) for every element, whole warps at a time, in no order
  const auto for_each = [&](const auto& f) {
    uint32_t t = 0;
    for (uint32_t i0 = 0; i0 < m; i0 += kChunk) {
      uint32_t k[kItems];
#pragma unroll
      for (uint32_t j = 0; j < kItems; ++j) {
        const uint32_t i = i0 + j * kBucketThreads + tid;
        k[j] = i < m ? src_k[src.seek(i, t)] : 0u;
      }
#pragma unroll
      for (uint32_t j = 0; j < kItems; ++j) f(k[j], i0 + j * kBucketThreads + tid < m);
    }
  };
  uint32_t pad_at = start;  // the padding run, after the elements below it
  if (pad.n) {
    if (tid == 0) sh.cnt[0] = 0u;
    __syncthreads();
    uint32_t L = 0;
    for_each([&](uint32_t k, bool ok) { L += ok && k < pad.kv ? 1u : 0u; });
    L = __reduce_add_sync(0xffffffffu, L);
    if (lane == 0) atomicAdd(&sh.cnt[0], L);
    __syncthreads();
    pad_at += sh.cnt[0];
  }
  KeyTurn turn;
  uint32_t done = 0;
  while (done < m) {
    const uint32_t a = turn.a, b = turn.b;
    // A key that may be hot: the most frequent one within a warp among 512
    // elements taken at even distances.
    __syncthreads();
    if (tid == 0) {
      sh.cnt[0] = sh.cnt[1] = sh.cnt[2] = 0u;
      sh.mn = 0xFFFFFFFFu;
      sh.mx = 0u;
    }
    const uint32_t one = src_k[src.find(uint32_t(uint64_t(tid) * m / kBucketThreads))];
    const bool has = one >= a && one <= b;
    const uint32_t peers = __match_any_sync(0xffffffffu, key_of(one)) & __ballot_sync(0xffffffffu, has);
    const uint32_t most = __reduce_max_sync(0xffffffffu, has ? (uint32_t(__popc(peers)) << 5) | lane : 0u);
    const uint32_t cand = __shfl_sync(0xffffffffu, key_of(one), int(most & 31u));
    if (lane == 0) {
      sh.cand[warp] = cand;
      sh.votes[warp] = most >> 5;
    }
    __syncthreads();
    uint32_t votes = 0, hot = 0;
    for (int w = 0; w < kBucketWarps; ++w)
      if (sh.votes[w] > votes) {
        votes = sh.votes[w];
        hot = sh.cand[w];
      }
    // the elements of [a, b]: how many, the range they span, how many below
    // the candidate key and of it
    uint32_t c = 0, mn = 0xFFFFFFFFu, mx = 0u, below = 0, copies = 0, tombs = 0;
    for_each([&](uint32_t k, bool ok) {
      if (ok && k >= a && k <= b) {
        ++c;
        mn = min(mn, k);
        mx = max(mx, k);
        below += key_of(k) < hot ? 1u : 0u;
        copies += key_of(k) == hot ? 1u : 0u;
        tombs += k == hot << 1 ? 1u : 0u;
      }
    });
    c = __reduce_add_sync(0xffffffffu, c);
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    below = __reduce_add_sync(0xffffffffu, below);
    copies = __reduce_add_sync(0xffffffffu, copies);
    tombs = __reduce_add_sync(0xffffffffu, tombs);
    if (lane == 0 && c) {
      atomicAdd(&sh.cnt[0], c);
      atomicMin(&sh.mn, mn);
      atomicMax(&sh.mx, mx);
      if (below) atomicAdd(&sh.cnt[1], below);
      if (copies) atomicAdd(&sh.cnt[2], copies);
    }
    if (lane == 0) sh.excl[warp] = tombs;
    __syncthreads();
    c = sh.cnt[0];
    mn = sh.mn;
    mx = sh.mx;
    below = sh.cnt[1];
    copies = sh.cnt[2];
    tombs = 0;
    for (int w = 0; w < kBucketWarps; ++w) tombs += sh.excl[w];
    if (c == 0) {  // (only below an upper part that is still to do)
      turn.next();
      continue;
    }
    if (mn == mx) {  // one key variable (the candidate may be another key)
      hot = key_of(mn);
      below = 0;
      copies = c;
      tombs = mn & 1u ? 0u : c;
    }
    if (c == m && c - copies > kMaxParts * kBucketCap) {
      __syncthreads();
      sort_digits(src_k, src_v, src, out_k + start, out_v + start, m, mn, mx, pad, bsm, sh);
      break;
    }
    if (c - copies > kBucketCap) {
      // Sub-bins over [mn, mx]; the lanes that share the sub-bin of the
      // warp's first active lane add their count at once (hot keys would
      // serialise the adds).
      const SubMap map = SubMap::of(mn, float(mx - mn) + 1.0f);
      __syncthreads();
      for (uint32_t i = tid; i < kSubBins; i += kBucketThreads) cnt[i] = 0u;
      if (tid == 0) sh.max = 0u;
      __syncthreads();
      for_each([&](uint32_t k, bool ok) {
        const uint32_t s = ok && k >= a && k <= b ? map.sub(k) : kSubBins;
        const uint32_t act = __ballot_sync(0xffffffffu, s < kSubBins);
        if (!act) return;
        const int lead = __ffs(int(act)) - 1;
        const uint32_t same = __ballot_sync(0xffffffffu, s == __shfl_sync(0xffffffffu, s, lead));
        if (int(lane) == lead) atomicAdd(&cnt[s], uint32_t(__popc(same)));
        else if (s < kSubBins && !((same >> lane) & 1u)) atomicAdd(&cnt[s], 1u);
      });
      __syncthreads();
      constexpr uint32_t kPer = kSubBins / kBucketThreads;
      uint32_t sum = 0;
      for (uint32_t e = 0; e < kPer; ++e) sum += cnt[tid * kPer + e];
      uint32_t all, fit = 0;  // sub-bins [0, fit) hold at most kBucketCap elements
      uint32_t run = block_excl_scan<kBucketThreads>(sum, sh.scan, all);
      for (uint32_t e = 0; e < kPer; ++e) {
        run += cnt[tid * kPer + e];
        if (run <= kBucketCap) fit = tid * kPer + e + 1;
      }
      if (fit) atomicMax(&sh.max, fit);
      __syncthreads();
      fit = sh.max;
      turn.narrow(mn, map, fit);
      continue;
    }
    if (c <= kBucketCap) copies = tombs = 0;  // all of them fit: no key is singled out
    // gather [a, b] in order: copies of the hot key to their places, the
    // rest to shared memory; a warp takes 256 consecutive elements
    uint32_t *ak = bsm, *av = bsm + kBucketCap;
    uint32_t kept = 0, dst0 = start + done + below + shift(hot << 1),
             dst1 = start + done + below + tombs + shift((hot << 1) | 1u), t = 0;
    const uint32_t lt = lanemask_lt();
    for (uint32_t c0 = 0; c0 < m; c0 += kChunk) {
      uint32_t k[kItems], v[kItems];
#pragma unroll
      for (uint32_t j = 0; j < kItems; ++j) {
        const uint32_t i = c0 + warp * (32 * kItems) + j * 32 + lane;
        const uint32_t at = i < m ? src.seek(i, t) : 0u;
        k[j] = i < m ? src_k[at] : 0u;
        v[j] = i < m ? src_v[at] : 0u;
      }
      // kind of element j of this lane, two bits: 0 outside [a, b], 1 to
      // shared memory, 2 a tombstone of the hot key, 3 a regular element of it
      uint32_t kind = 0, n1 = 0, n2 = 0, n3 = 0;
#pragma unroll
      for (uint32_t j = 0; j < kItems; ++j) {
        const bool in = c0 + warp * (32 * kItems) + j * 32 + lane < m && k[j] >= a && k[j] <= b;
        const uint32_t x = !in ? 0u : (copies && key_of(k[j]) == hot ? 2u + (k[j] & 1u) : 1u);
        kind |= x << (2 * j);
        const uint32_t lo = __ballot_sync(0xffffffffu, x & 1u), hi = __ballot_sync(0xffffffffu, x & 2u);
        n1 += __popc(lo & ~hi);
        n2 += __popc(hi & ~lo);
        n3 += __popc(lo & hi);
      }
      __syncthreads();
      if (lane == 0) sh.cand[warp] = n1 | (n2 << 10) | (n3 << 20);
      __syncthreads();
      uint32_t p1 = kept, p2 = dst0, p3 = dst1;
      for (uint32_t w = 0; w < uint32_t(kBucketWarps); ++w) {
        const uint32_t x = sh.cand[w];
        const bool before = w < warp;
        p1 += before ? x & 1023u : 0u;
        p2 += before ? (x >> 10) & 1023u : 0u;
        p3 += before ? x >> 20 : 0u;
        kept += x & 1023u;
        dst0 += (x >> 10) & 1023u;
        dst1 += x >> 20;
      }
#pragma unroll
      for (uint32_t j = 0; j < kItems; ++j) {
        const uint32_t x = (kind >> (2 * j)) & 3u;
        const uint32_t lo = __ballot_sync(0xffffffffu, x & 1u), hi = __ballot_sync(0xffffffffu, x & 2u);
        const uint32_t mask = (x & 1u ? lo : ~lo) & (x & 2u ? hi : ~hi);
        const uint32_t at = (x == 1u ? p1 : (x == 2u ? p2 : p3)) + __popc(mask & lt);
        if (x == 1u) {
          ak[at] = k[j];
          av[at] = v[j];
        } else if (x) {
          out_k[at] = k[j];
          out_v[at] = v[j];
        }
        p1 += __popc(lo & ~hi);
        p2 += __popc(hi & ~lo);
        p3 += __popc(lo & hi);
      }
    }
    __syncthreads();
    if (kept) {
      const BucketRange part{mn, mx, SubMap::of(mn, float(mx - mn) + 1.0f)};
      const auto load = [&](uint32_t (&kv)[kBucketIPT], uint32_t (&v)[kBucketIPT]) {
#pragma unroll
        for (int j = 0; j < kBucketIPT; ++j) {
          const uint32_t i = tid + j * kBucketThreads;
          if (i < kept) {
            kv[j] = ak[i];
            v[j] = av[i];
          }
        }
      };
      sort_resident<true>(load, kept, part, bsm, sh, [&](uint32_t i, uint32_t kk, uint32_t vv) {
        const uint32_t dst = start + done + i + (copies && key_of(kk) > hot ? copies : 0u) + shift(kk);
        out_k[dst] = kk;
        out_v[dst] = vv;
      });
    }
    done += c;
    turn.next();
  }
  __syncthreads();  // (the passes use the padding's places)
  for (uint32_t j = tid; j < pad.n; j += kBucketThreads) {
    out_k[pad_at + j] = pad.kv;
    out_v[pad_at + j] = pad.v;
  }
  __syncthreads();  // the caller reads the output back
}

// Prefix-index entries `bins` of a bucket at `start`: the elements in `view`
// and the padding run.  `ends`: bit 0 when the bucket holds the first element
// of the output, bit 1 the last; its entries are then written inside the
// populated bin range only, whose bound is recorded.
__device__ __forceinline__ void write_bins(const SortedView& view, uint32_t start, const PadRun& pad, BinRange bins,
                                           int ends) {
  if (!bins.fence) return;
  if (ends) {
    const uint32_t nb = fence_bins(bins.fshift);
    if (ends & 1) {
      const uint32_t kv = min(view.m ? view.smallest() : pad.kv, pad.n ? pad.kv : 0xFFFFFFFFu);
      bins.bin0 = max(bins.bin0, fence_bin(kv, bins.fshift) + 1);
      if (threadIdx.x == 0) bins.fence[nb + 2] = fence_bin(kv, bins.fshift);
    }
    if (ends & 2) {
      const uint32_t kv = max(view.m ? view.largest() : pad.kv, pad.n ? pad.kv : 0u);
      bins.bin1 = min(bins.bin1, fence_bin(kv, bins.fshift) + 1);
      if (threadIdx.x == 0) {
        bins.fence[nb + 3] = fence_bin(kv, bins.fshift);
        bins.fence[nb] = start + view.m + pad.n;
      }
    }
  }
  for (uint32_t P = bins.bin0 + threadIdx.x; P < bins.bin1; P += blockDim.x) {
    const uint32_t kv = P << bins.fshift;
    bins.fence[P] = start + (view.m ? view.less(kv) : 0u) + (pad.n && kv > pad.kv ? pad.n : 0u);
  }
}

// A bucket that fits shared memory: the elements given by `load` (see
// sort_resident), with the padding run at its sorted place, to out[start ..)
// and its prefix-index entries.
// With kMaySkip, out_k null writes the bins alone.
template <bool kMaySkip = false, class Load>
__device__ __forceinline__ void resident_body(const Load& load, uint32_t* out_k, uint32_t* out_v, uint32_t start,
                                              uint32_t m, const BucketRange& range, const PadRun& pad,
                                              const BinRange& bins, int ends, uint32_t* bsm, BucketShared& sh) {
  SortedView view{bsm, 0u, nullptr, range.map};
  if (m)
    view = sort_resident<false>(load, m, range, bsm, sh, [&](uint32_t i, uint32_t k, uint32_t v) {
      if (kMaySkip && !out_k) return;
      const uint32_t dst = start + i + (pad.n && k >= pad.kv ? pad.n : 0u);
      out_k[dst] = k;
      out_v[dst] = v;
    });
  if (pad.n && !(kMaySkip && !out_k)) {
    const uint32_t L = m ? view.less(pad.kv) : 0u;
    for (uint32_t j = threadIdx.x; j < pad.n; j += blockDim.x) {
      out_k[start + L + j] = pad.kv;
      out_v[start + L + j] = pad.v;
    }
  }
  write_bins(view, start, pad, bins, ends);
}

// One bucket, one CTA of kBucketThreads: sorts the m elements src.at(0 ..
// m - 1) of (src_k, src_v) stably by the key variable into out[start, start +
// m + pad.n) and writes the prefix-index entries `bins` of the result.  The
// padding run (a short batch's, which comes first among equal key variables
// in the stable order) is written at its sorted place.
template <class Src>
__device__ __forceinline__ void bucket_body(uint32_t* src_k, uint32_t* src_v, const Src& src,
                                            uint32_t* out_k, uint32_t* out_v, uint32_t start, uint32_t m,
                                            const BucketRange& range, const PadRun& pad, BinRange bins, int ends,
                                            uint32_t* bsm, BucketShared& sh) {
  SortedView view{out_k + start, m + pad.n, nullptr, range.map};
  if (m > kBucketCap) {
    sort_big(src_k, src_v, src, out_k, out_v, start, m, range, pad, bsm, sh);
    write_bins(view, start, PadRun{0u, 0u, 0u}, bins, ends);
    return;
  }
  const auto load = [&](uint32_t (&kv)[kBucketIPT], uint32_t (&v)[kBucketIPT]) {
#pragma unroll
    for (int j = 0; j < kBucketIPT; ++j) {
      const uint32_t i = threadIdx.x + j * kBucketThreads;
      if (i < m) {
        const uint32_t at = src.at(i);
        kv[j] = __ldg(src_k + at);  // (sort_digits of other buckets writes their own places only)
        v[j] = __ldg(src_v + at);
      }
    }
  };
  resident_body(load, out_k, out_v, start, m, range, pad, bins, ends, bsm, sh);
}

// A batch whose deferred key check failed becomes n placebo tombstones (the
// key 2^31 - 1 that no query sees), all in the last bin.  CTA d of `ctas`.
__device__ __forceinline__ void write_placebos(uint32_t* out_k, uint32_t* out_v, uint32_t n, uint32_t* fence,
                                               int fshift, uint32_t d, uint32_t ctas) {
  const uint32_t at = d * blockDim.x + threadIdx.x, step = ctas * blockDim.x;
  for (uint32_t i = at; i < n; i += step) {
    out_k[i] = kPlaceboKv;
    out_v[i] = 0u;
  }
  if (fence) {
    const uint32_t nb = fence_bins(fshift);
    for (uint32_t i = at; i < nb; i += step) fence[i] = 0u;
    if (at == 0) {
      fence[nb] = n;
      fence[nb + 2] = 0u;
      fence[nb + 3] = nb - 1;
    }
  }
}

// The whole sort of at most kBucketCap elements in one launch: bound by the
// chain of its barriers, 4.1 us where the two kernels took 12.2
// (lsm_sort_pairs of 2^10 pairs, back to back).  CTA 0 alone writes the sorted
// elements; with a prefix index, which has 2^16 entries or more however small
// the batch, every CTA of the grid sorts the batch and writes its share of the
// entries.  (Update calls of 1051 / 5000 uniform keys: 28.8 / 39.8 us with all
// entries written by one CTA, now 10.4 / 10.7; the two kernels 19.6 / 21.1.
// Between 512 and 16384 entries a CTA the calls differ by their spread only:
// 15.2 .. 16.4 and 16.4 .. 17.1 us with a reset in the loop.)
constexpr uint32_t kSmallBins = 2048;  // entries per CTA
__global__ void __launch_bounds__(kBucketThreads) small_sort(Loader ld, uint32_t* out_k, uint32_t* out_v,
                                                             uint32_t* fence, int fshift, uint32_t* host,
                                                             uint32_t seq, uint32_t* defer_err) {
  extern __shared__ __align__(16) uint32_t bsm[];
  __shared__ BucketShared sh;
  pdl_trigger();
  pdl_wait();
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t npad = ld.npad(), m = ld.n - npad;
  uint32_t kv[kBucketIPT], v[kBucketIPT];
  bool bad = false;
  ld.load_items(npad + tid, uint32_t(kBucketThreads), [&](uint32_t p) { return p < ld.n; }, kv, v, bad);
  uint32_t mn = 0xFFFFFFFFu, mx = 0u;
#pragma unroll
  for (int j = 0; j < kBucketIPT; ++j) {
    if (tid + j * kBucketThreads < m) {
      mn = min(mn, kv[j]);
      mx = max(mx, kv[j]);
    }
  }
  mn = __reduce_min_sync(0xffffffffu, mn);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) {
    sh.cand[warp] = mn;
    sh.votes[warp] = mx;
  }
  const int any_bad = __syncthreads_or(bad);
  if (tid == 0 && host && blockIdx.x == 0) *reinterpret_cast<volatile uint32_t*>(host) = check_word(seq, any_bad != 0);
  if (any_bad && defer_err) {
    write_placebos(out_k, out_v, ld.n, fence, fshift, blockIdx.x, gridDim.x);
    if (tid == 0 && blockIdx.x == 0) atomicOr(defer_err, kErrBadKey);
    return;
  }
  const uint32_t w = lane & uint32_t(kBucketWarps - 1);
  mn = __reduce_min_sync(0xffffffffu, sh.cand[w]);
  mx = __reduce_max_sync(0xffffffffu, sh.votes[w]);
  PadRun pad{npad, 0u, 0u};
  if (npad) ld.load(0, pad.kv, pad.v, bad);
  const uint32_t share = fence ? fence_bins(fshift) / gridDim.x : 0u;
  const BinRange bins{fence, fshift, blockIdx.x * share, (blockIdx.x + 1) * share};
  if (blockIdx.x) out_k = nullptr;
  const BucketRange range{mn, mx, SubMap::of(mn, float(mx - mn) + 1.0f)};
  const auto load = [&](uint32_t (&k)[kBucketIPT], uint32_t (&x)[kBucketIPT]) {
#pragma unroll
    for (int j = 0; j < kBucketIPT; ++j) {
      k[j] = kv[j];
      x[j] = v[j];
    }
  };
  resident_body<true>(load, out_k, out_v, 0u, m, range, pad, bins, 3, bsm, sh);
}

__global__ void __launch_bounds__(kBucketThreads, 2) bucket_sort(Loader ld, uint32_t* tmp_k, uint32_t* tmp_v,
                                                              const uint2* __restrict__ runs, uint32_t* out_k,
                                                              uint32_t* out_v, const uint32_t* __restrict__ ctl,
                                                              uint32_t n, uint32_t* fence, int fshift,
                                                              uint32_t* __restrict__ next_ctl,
                                                              uint32_t* defer_err) {
  extern __shared__ __align__(16) uint32_t bsm[];
  __shared__ BucketShared sh;
  __shared__ uint32_t s_rstart[kMsdMaxTiles + 1], s_rbase[kMsdMaxTiles];
  __shared__ uint8_t s_chunk[kBucketCap / 16];
  pdl_trigger();
  pdl_wait();
  const uint32_t tid = threadIdx.x, d = blockIdx.x;
  const uint32_t ntiles = (n + kMsdTile - 1) / kMsdTile;
  // the control block of the next sort starts zeroed (it is idle now)
  if (d == 0)
    for (uint32_t i = tid; i < uint32_t(kSortCtlWords); i += kBucketThreads) next_ctl[i] = 0u;
  if (defer_err && ctl[kSortCtlStatus]) {
    write_placebos(out_k, out_v, n, fence, fshift, d, kRadix);
    if (d == 0 && tid == 0) atomicOr(defer_err, kErrBadKey);
    return;
  }
  // this bucket's run in every tile, in tile order, and the buckets' totals
  // (one round trip); one scan for the runs' starts and the sum of the totals
  // before the bucket, its start in the output
  const uint2 run = tid < ntiles ? runs[d * kMsdMaxTiles + tid] : make_uint2(0u, 0u);
  const uint32_t before = tid < d ? ctl[3 * kRadix + tid] : 0u;
  const uint32_t map_lo = ctl[kSortCtlMap], map_mul = ctl[kSortCtlMap + 1];
  const bool top = d == kRadix - 1;
  const uint32_t lo = ctl[kSortCtlBounds + d], next = top ? 0xFFFFFFFFu : ctl[kSortCtlBounds + d + 1];
  const uint32_t hi = next == 0xFFFFFFFFu ? next : next - 1;
  uint64_t sums;
  const uint64_t own = run.y | (uint64_t(before) << 32);
  const uint32_t rs = uint32_t(block_excl_scan<kBucketThreads, uint64_t>(own, sh.scan64, sums));
  const uint32_t m = uint32_t(sums), start = uint32_t(sums >> 32);
  if (tid < ntiles) {
    s_rstart[tid] = rs;
    s_rbase[tid] = run.x - rs;
    // the chunks (16 elements) whose first element lies in this run
    if (m <= kBucketCap)
      for (uint32_t c = (rs + 15) >> 4; c < ((rs + run.y + 15) >> 4); ++c) s_chunk[c] = uint8_t(tid);
  }
  if (tid == 0) s_rstart[ntiles] = m;
  __syncthreads();
  // a short batch's padding: one run in the bucket of its key variable
  PadRun pad{ld.npad(), 0u, 0u};
  if (pad.n) {
    bool bad;
    ld.load(0, pad.kv, pad.v, bad);
    if (pad.kv < lo || pad.kv > hi || hi < lo) pad.n = 0;
  }
  const uint32_t total = m + pad.n;
  // An empty bucket writes its bins too (they share the next element's
  // position), unless nothing comes before or after it.
  if (total == 0 && (start == 0 || start == n)) return;
  BinRange bins{fence, fshift, 0u, 0u};
  if (fence) {
    bins.bin0 = d ? ((lo - 1) >> fshift) + 1 : 0u;
    bins.bin1 = (hi >> fshift) + 1;
  }
  // keys below the sampled range (bucket 0) and above it (bucket 255) share
  // the sub-bins at that end
  const BucketRange range{lo, hi, SubMap::of(d ? lo : map_lo, __fdividef(4294967296.0f, float(map_mul)) + 1.0f)};
  const int ends = (total && start == 0 ? 1 : 0) | (total && start + total == n ? 2 : 0);
  const RunSrc src{s_rstart, s_rbase, s_chunk, ntiles};
  bucket_body(tmp_k, tmp_v, src, out_k, out_v, start, m, range, pad, bins, ends, bsm, sh);
}

__global__ void __launch_bounds__(256) check_keys(const uint32_t* __restrict__ keys, uint64_t n,
                                                  uint32_t* status) {
  bool bad = false;
  for (uint64_t i = blockIdx.x * 256ull + threadIdx.x; i < n; i += uint64_t(gridDim.x) * 256ull)
    bad |= __ldg(keys + i) > kMaxUserKey;
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, kErrBadKey);
}

// ---------------------------------------------------------------------------
// The batch sort of the batched form: the same bucket scheme on every
// instance's batch at once.  Instance i splits the key range of its batch, by
// 512 samples of it that every CTA of mseg_count reads, in 2^d_i parts of about
// 4096 elements (PartMap; without hot keys); its batch is cut into
// kMultiSortTile-element tiles; one launch per phase covers every tile or
// bucket of every instance.  Instances without a batch this round (count 0,
// or refused by the prep kernel) leave at once.
// ---------------------------------------------------------------------------
constexpr int kMultiIPT = int(kMultiSortTile) / kThreads;  // 16
static_assert(kMultiIPT * kThreads == int(kMultiSortTile), "tile");
static_assert(kScatterIPT * kScatterThreads == int(kMultiSortTile), "tile");

__device__ __forceinline__ uint32_t multi_ops(const MultiBatch& in, const MultiInst& d, uint32_t i) {
  return in.counts ? __ldg(in.counts + i) : d.b;
}

// Elements p0 + step j, j < N, below m of the tile at t0 of an instance's
// reversed padded batch (element p is op min(b - 1 - p, nops - 1)): all loads
// are issued before the first is used.  Elements outside keep kv = v = 0.
// (One element after another, its value once its key had come, and 16 a thread
// in mseg_scatter instead of 8: eight rounds of 128 dictionaries, 2^10 to 2^18
// operations each, took 4042 us; now 3617.)
template <bool kVals, int N>
__device__ __forceinline__ void multi_load_items(const MultiBatch& in, const MultiInst& d, uint32_t nops, uint32_t t0,
                                                 uint32_t m, uint32_t p0, uint32_t step, uint32_t (&kv)[N],
                                                 uint32_t (&v)[N], bool& bad) {
  const uint32_t last = d.b - 1 - t0;
  const uint32_t* keys = in.keys + d.in_off;
  const uint32_t* vals = in.vals + d.in_off;
  const uint8_t* del = in.del + d.in_off;
  uint32_t fl[N];
  const auto load = [&](auto with_del, auto with_vals) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const uint32_t p = p0 + j * step;
      kv[j] = v[j] = fl[j] = 0u;
      if (p < m) {
        const uint32_t s = min(last - p, nops - 1);
        kv[j] = __ldg(keys + s);
        if (decltype(with_del)::value) fl[j] = __ldg(del + s);
        if (decltype(with_vals)::value) v[j] = __ldg(vals + s);
      }
    }
  };
  const bool has_vals = kVals && in.vals;
  if (in.del && has_vals) load(std::true_type{}, std::true_type{});
  else if (in.del) load(std::true_type{}, std::false_type{});
  else if (has_vals) load(std::false_type{}, std::true_type{});
  else load(std::false_type{}, std::false_type{});
#pragma unroll
  for (int j = 0; j < N; ++j) {
    if (p0 + j * step >= m) continue;
    const bool b = kv[j] > kMaxUserKey;
    bad |= b;
    kv[j] = b ? kPlaceboKv : ((kv[j] << 1) | (fl[j] ? 0u : 1u));
    if (!(kv[j] & 1u)) v[j] = 0u;
  }
}

__global__ void __launch_bounds__(kThreads) mseg_count(MultiArena ar, MultiBatch in) {
  __shared__ uint32_t s_h[kRadix], s_mn[kWarps], s_mx[kWarps];
  const uint32_t tid = threadIdx.x, gt = blockIdx.x;
  const uint32_t i = find_instance_warp(ar.stile_prefix, ar.n, gt);
  const MultiInst& d = ar.inst[i];
  const uint32_t nops = multi_ops(in, d, i);
  if (nops == 0 || nops > d.b) return;  // whole CTA: no batch, or refused
  s_h[tid] = 0;
  const uint32_t t0 = (gt - d.stile0) * kMultiSortTile;
  const uint32_t m = (d.b - t0) < kMultiSortTile ? (d.b - t0) : kMultiSortTile;
  bool bad_any = false;
  uint32_t kv[kMultiIPT], v[kMultiIPT], sample[2];
#pragma unroll
  for (uint32_t e = 0; e < 2; ++e)
    sample[e] = __ldg(in.keys + d.in_off + uint32_t(uint64_t(2 * tid + e) * nops / (2 * kThreads)));
  multi_load_items<false>(in, d, nops, t0, m, tid, uint32_t(kThreads), kv, v, bad_any);
#pragma unroll
  for (uint32_t e = 0; e < 2; ++e)
    sample[e] = sample[e] > kMaxUserKey ? kPlaceboKv : (sample[e] << 1) | 1u;
  const uint32_t mn = __reduce_min_sync(0xffffffffu, min(sample[0], sample[1])),
                 mx = __reduce_max_sync(0xffffffffu, max(sample[0], sample[1]));
  if (lane_id() == 0) {
    s_mn[tid >> 5] = mn;
    s_mx[tid >> 5] = mx;
  }
  __syncthreads();
  const uint32_t w = lane_id() & uint32_t(kWarps - 1);
  const PartMap map = PartMap::spanning(__reduce_min_sync(0xffffffffu, s_mn[w]),
                                        __reduce_max_sync(0xffffffffu, s_mx[w]), d.msd_bits);
  if (t0 == 0 && tid == 0) {
    ar.map[2 * i] = map.fine.lo;
    ar.map[2 * i + 1] = map.fine.mul;
  }
#pragma unroll
  for (int j = 0; j < kMultiIPT; ++j)
    if (j * kThreads + tid < m) atomicAdd(&s_h[map.part(kv[j])], 1u);
  const int any_bad = __syncthreads_or(bad_any);
  ar.tilecnt[uint64_t(gt) * 512 + tid] = s_h[tid];
  if (any_bad && tid == 0) atomicOr(ar.badkey + i, 1u);
}

// Per instance (one CTA, thread = bucket): where each tile's run of each
// bucket goes, relative to the instance's batch start.
__global__ void __launch_bounds__(kThreads) mseg_offsets(MultiArena ar) {
  __shared__ uint32_t s_scan[kWarps];
  const uint32_t i = blockIdx.x, tid = threadIdx.x;
  if (ar.k[i] < 0) return;
  const MultiInst& d = ar.inst[i];
  const uint32_t nbk = 1u << d.msd_bits;
  const uint32_t ntiles = (d.b + kMultiSortTile - 1) / kMultiSortTile;
  uint32_t* tc = ar.tilecnt + uint64_t(d.stile0) * 512;
  uint32_t total = 0;
  if (tid < nbk)
    for (uint32_t t = 0; t < ntiles; ++t) total += tc[t * 512 + tid];
  uint32_t all;
  const uint32_t start = block_excl_scan<kThreads>(total, s_scan, all);
  if (tid < nbk) {
    uint32_t run = start;
    for (uint32_t t = 0; t < ntiles; ++t) {
      const uint32_t c = tc[t * 512 + tid];
      tc[t * 512 + 256 + tid] = run;
      run += c;
    }
    ar.bstart[d.bucket0 + tid] = start;
    ar.bcnt[d.bucket0 + tid] = total;
    const PartMap map = PartMap::of(ar.map[2 * i], ar.map[2 * i + 1], d.msd_bits);
    ar.blo[d.bucket0 + tid] = tid ? map.lower(tid) : 0u;
  }
}

__global__ void __launch_bounds__(kScatterThreads) mseg_scatter(MultiArena ar, MultiBatch in) {
  __shared__ __align__(16) uint32_t s_keys[kMultiSortTile];
  __shared__ __align__(16) uint32_t s_vals[kMultiSortTile];
  __shared__ uint32_t s_whist[kScatterWarps][kRadix];
  __shared__ uint32_t s_excl[kRadix], s_gbase[kRadix], s_scan[kScatterWarps];
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, gt = blockIdx.x;
  const uint32_t i = find_instance_warp(ar.stile_prefix, ar.n, gt);
  if (ar.k[i] < 0) return;  // whole CTA
  const MultiInst& d = ar.inst[i];
  const uint32_t nops = multi_ops(in, d, i);
  const uint32_t t0 = (gt - d.stile0) * kMultiSortTile;
  const uint32_t m = (d.b - t0) < kMultiSortTile ? (d.b - t0) : kMultiSortTile;
  const PartMap map = PartMap::of(ar.map[2 * i], ar.map[2 * i + 1], d.msd_bits);
  const uint32_t base = warp * (32 * kScatterIPT);
  uint32_t kv[kScatterIPT], v[kScatterIPT], rank[kScatterIPT];
  bool bad_any = false;  // (mseg_count has seen them)
  multi_load_items<true>(in, d, nops, t0, m, base + lane, 32u, kv, v, bad_any);
  if (tid < kRadix) s_gbase[tid] = ar.tilecnt[uint64_t(gt) * 512 + 256 + tid];
  rank_block<kScatterThreads, kScatterIPT>(kv, m, base, [&](uint32_t k) { return map.part(k); }, rank, s_whist,
                                           s_excl, s_scan, nullptr);
#pragma unroll
  for (int j = 0; j < kScatterIPT; ++j) {
    const uint32_t p = base + j * 32 + lane;
    if (p < m) {
      const uint32_t dg = map.part(kv[j]);
      const uint32_t pos = s_excl[dg] + s_whist[warp][dg] + rank[j];
      s_keys[pos] = kv[j];
      s_vals[pos] = v[j];
    }
  }
  __syncthreads();
  uint32_t* tk = ar.tkeys + d.boff;
  uint32_t* tv = ar.tvals + d.boff;
  for (uint32_t e = tid; e < m; e += kScatterThreads) {
    const uint32_t k = s_keys[e];
    const uint32_t dg = map.part(k);
    const uint32_t dst = s_gbase[dg] + (e - s_excl[dg]);
    if (dst < d.b) {
      tk[dst] = k;
      tv[dst] = s_vals[e];
    }
  }
}

// One bucket of one instance per CTA: sorted into level 0 (when the round's
// fold target is level 0) or the sorted-batch buffer, with that run's
// prefix-index entries.  With the top d bits as the bucket, keys below 2^26 all
// fell in one: eight rounds of 10 dictionaries of up to 27181 operations took
// 2214 us, now 479; keys below 2^30 (85 dictionaries, seven rounds) 1443 and
// 588; over the whole key range the samples cost 0.5 % (128 dictionaries 3619
// and 3637 us).
__global__ void __launch_bounds__(kBucketThreads, 2) mseg_bucket(MultiArena ar) {
  extern __shared__ __align__(16) uint32_t bsm[];
  __shared__ BucketShared sh;
  const uint32_t gb = blockIdx.x;
  const uint32_t i = find_instance_warp(ar.bucket_prefix, ar.n, gb);
  const int k = ar.k[i];
  if (k < 0) return;  // whole CTA
  const MultiInst& d = ar.inst[i];
  const uint32_t bucket = gb - d.bucket0;
  const uint32_t start = ar.bstart[gb], m = ar.bcnt[gb];
  uint32_t *ok, *ov, *of;
  if (k == 0) {
    ok = ar.keys + d.lvl_off[0];
    ov = ar.vals + d.lvl_off[0];
    of = ar.fence + d.lvl_fence[0];
  } else {
    ok = ar.bkeys + d.boff;
    ov = ar.bvals + d.boff;
    of = ar.fence + d.batch_fence;
  }
  const int fs = d.fshift0;
  uint32_t* tk = ar.tkeys + d.boff;
  uint32_t* tv = ar.tvals + d.boff;
  const bool top = bucket == (1u << d.msd_bits) - 1;
  const uint32_t lo = ar.blo[gb], next = top ? 0xFFFFFFFFu : ar.blo[gb + 1];
  const uint32_t hi = next == 0xFFFFFFFFu ? next : next - 1;
  const BucketRange range{lo, hi, SubMap::of(bucket ? lo : ar.map[2 * i], PartMap::width(ar.map[2 * i + 1], d.msd_bits))};
  const BinRange bins{of, fs, bucket ? ((lo - 1) >> fs) + 1 : 0u, (hi >> fs) + 1};
  bucket_body(tk, tv, ContigSrc{start}, ok, ov, start, m, range, PadRun{0u, 0u, 0u}, bins, 0, bsm, sh);
  if (top && threadIdx.x == 0) {
    const uint32_t nb = fence_bins(fs);
    of[nb] = d.b;
    of[nb + 2] = 0u;
    of[nb + 3] = nb - 1;
  }
}

}  // namespace

constexpr size_t kBucketSmem = 4 * size_t(kBucketCap) * sizeof(uint32_t) + size_t(kBucketCap) * sizeof(uint16_t);
PerDeviceFlags g_bucket_attr[2], g_pass_attr[2];

cudaError_t bucket_sort_launch(const SortArgs& a, SortWorkspace& ws, cudaStream_t st, uint32_t* status,
                               uint32_t seq) {
  cudaError_t e;
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = set_smem_attr_once(bucket_sort, kBucketSmem, dev, g_bucket_attr[0])) != cudaSuccess) return e;
  const uint32_t ntiles = (a.n + kMsdTile - 1) / kMsdTile;
  uint2* runs = reinterpret_cast<uint2*>(ws.tilecnt);
  uint32_t* ctl = ws.ctl + ws.flip * kSortCtlWords;
  uint32_t* next = ws.ctl + (ws.flip ^ 1) * kSortCtlWords;
  Loader ld{a.mode, a.in_keys, a.in_vals, a.in_del, uint32_t(a.n_in), a.n};
  // a deferred check leaves its verdict in the sort's own control block
  const KeyCheck check{a.defer_err ? nullptr : status, seq, a.defer_err || status};
  if (a.n <= kBucketCap) {
    if ((e = set_smem_attr_once(small_sort, kBucketSmem, dev, g_bucket_attr[1])) != cudaSuccess) return e;
    count_launches(1);  // (the control block stays as it is)
    // (a sort without a prefix index may be in place: one CTA)
    const uint32_t ctas = a.fence ? max(1u, min(fence_bins(a.fshift) / kSmallBins, 128u)) : 1u;
    return launch_pdl(small_sort, dim3(ctas), dim3(kBucketThreads), kBucketSmem, st, ld, a.out_keys, a.out_vals, a.fence,
                      a.fshift, a.defer_err ? nullptr : status, seq, a.defer_err);
  }
  count_launches(1);
  if ((e = launch_pdl(msd_tile, dim3(ntiles), dim3(kScatterThreads), 0, st, ld, a.tmp_keys, a.tmp_vals, runs, ctl,
                      check)) != cudaSuccess)
    return e;
  count_launches(1);
  if ((e = launch_pdl(bucket_sort, dim3(kRadix), dim3(kBucketThreads), kBucketSmem, st, ld,
                      a.tmp_keys, a.tmp_vals, static_cast<const uint2*>(runs), a.out_keys, a.out_vals,
                      static_cast<const uint32_t*>(ctl), a.n, a.fence, a.fshift, next, a.defer_err)) != cudaSuccess)
    return e;
  ws.flip ^= 1;
  return cudaSuccess;
}

cudaError_t sort_launch(const SortArgs& a, SortWorkspace& ws, cudaStream_t st, uint32_t* status, uint32_t seq) {
  if (a.n == 0) return cudaSuccess;
  if (a.n <= kMsdMaxN && ws.tilecnt) return bucket_sort_launch(a, ws, st, status, seq);
  const uint32_t ntiles = (a.n + kSortTile - 1) / kSortTile;
  if (ntiles > ws.max_tiles) return cudaErrorInvalidValue;
  cudaError_t e;
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = set_smem_attr_once(sort_pass<true>, kPassSmem, dev, g_pass_attr[0])) != cudaSuccess) return e;
  if ((e = set_smem_attr_once(sort_pass<false>, kPassSmem, dev, g_pass_attr[1])) != cudaSuccess) return e;
  if (++ws.epoch >= (1u << 30)) {
    ws.epoch = 1;
    e = cudaMemsetAsync(ws.lookback, 0, sizeof(uint64_t) * kSortPasses * ws.max_tiles * kRadix, st);
    if (e != cudaSuccess) return e;
  }
  uint32_t* ctl = ws.ctl + ws.flip * kSortCtlWords;
  e = cudaMemsetAsync(ctl, 0, sizeof(uint32_t) * kSortCtlWords, st);
  if (e != cudaSuccess) return e;
  Loader ld{a.mode, a.in_keys, a.in_vals, a.in_del, uint32_t(a.n_in), a.n};
  uint32_t hblocks = (a.n + kHistChunk - 1) / kHistChunk;
  if (hblocks > 4 * 152) hblocks = 4 * 152;
  count_launches(1);
  sort_histogram<<<hblocks, kPassThreads, 0, st>>>(ld, ctl, KeyCheck{status, seq, status != nullptr});
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // in -> tmp -> out -> tmp -> out
  uint32_t* bk[2] = {a.tmp_keys, a.out_keys};
  uint32_t* bv[2] = {a.tmp_vals, a.out_vals};
  const size_t lb_stride = size_t(ws.max_tiles) * kRadix;
  count_launches(1);
  sort_pass<true><<<ntiles, kPassThreads, kPassSmem, st>>>(ld, nullptr, nullptr, bk[0], bv[0], ctl, ws.lookback,
                                                0, ws.epoch, ws.sticky);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  for (int p = 1; p < kSortPasses; ++p) {
    count_launches(1);
    sort_pass<false><<<ntiles, kPassThreads, kPassSmem, st>>>(ld, bk[(p - 1) & 1], bv[(p - 1) & 1], bk[p & 1],
                                                   bv[p & 1], ctl, ws.lookback + p * lb_stride, p,
                                                   ws.epoch, ws.sticky);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  // leave the next half zeroed, as the bucket path does
  ws.flip ^= 1;
  e = cudaMemsetAsync(ws.ctl + ws.flip * kSortCtlWords, 0, sizeof(uint32_t) * kSortCtlWords, st);
  if (e != cudaSuccess) return e;
  if (a.fence) return build_fence_launch(a.out_keys, a.n, a.fence, a.fshift, st);
  return cudaSuccess;
}

cudaError_t check_keys_launch(const uint32_t* keys, uint64_t n, uint32_t* status, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  uint64_t blocks = (n + 255) / 256;
  if (blocks > 8 * 152) blocks = 8 * 152;
  count_launches(1);
  check_keys<<<unsigned(blocks), 256, 0, st>>>(keys, n, status);
  return cudaGetLastError();
}


cudaError_t multi_sort_count_launch(const MultiArena& ar, const MultiBatch& in, cudaStream_t st) {
  if (ar.total_stiles == 0) return cudaSuccess;
  count_launches(1);
  mseg_count<<<unsigned(ar.total_stiles), kThreads, 0, st>>>(ar, in);
  return cudaGetLastError();
}

cudaError_t multi_sort_prepare() {
  return cudaFuncSetAttribute(mseg_bucket, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kBucketSmem));
}

cudaError_t multi_sort_launch(const MultiArena& ar, const MultiBatch& in, cudaStream_t st) {
  cudaError_t e;
  if (ar.total_stiles == 0) return cudaSuccess;
  count_launches(1);
  mseg_offsets<<<ar.n, kThreads, 0, st>>>(ar);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  count_launches(1);
  mseg_scatter<<<unsigned(ar.total_stiles), kScatterThreads, 0, st>>>(ar, in);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  count_launches(1);
  mseg_bucket<<<unsigned(ar.total_buckets), kBucketThreads, kBucketSmem, st>>>(ar);
  return cudaGetLastError();
}

}  // namespace gpulsm

// ---------------------------------------------------------------------------
// Allocation-free batch sort (lsm_sort_pairs_noalloc in gpulsm.h).
//
// Some callers may not allocate device memory once they are running: a
// process whose memory is handed out by its own pool allocator and forbids
// raw cudaMalloc, or a latency-bound loop that cannot afford the implicit
// device-wide synchronisation and the unbounded time a cudaMalloc/cudaFree
// may take.  For them the sort below takes all of its scratch (the
// bucket sort's tile scratch, control words and run table) from
// one fixed array with static storage in this file, which every GPU that
// loads the library holds until the process exits.  Its size is set by
// kNoAllocMaxPairs.
// ---------------------------------------------------------------------------
#include <mutex>

#include "gpulsm.h"

namespace gpulsm {
namespace {

constexpr uint32_t kNoAllocMaxPairs = LSM_SORT_NOALLOC_MAX_PAIRS;
// Up to kMsdMaxN pairs the sort is the two-kernel bucket sort, which needs
// no look-back words; the array below holds only what that path uses.
static_assert(kNoAllocMaxPairs <= kMsdMaxN, "the allocation-free sort stays on the bucket path");
constexpr size_t kNoAllocCtl = 2112;                    // > 2 * kSortCtlWords, multiple of 64
constexpr size_t kNoAllocSticky = kNoAllocCtl - 1;      // last ctl word: device error bits
constexpr size_t kNoAllocTmpK = kNoAllocCtl;
constexpr size_t kNoAllocTmpV = kNoAllocTmpK + kNoAllocMaxPairs;
constexpr size_t kNoAllocRuns = kNoAllocTmpV + kNoAllocMaxPairs;  // run table
constexpr size_t kNoAllocWords = kNoAllocRuns + kMsdRunWords;
static_assert(kNoAllocCtl > 2 * size_t(kSortCtlWords), "both control halves and the error word fit");
static_assert(kNoAllocRuns % 2 == 0, "the run table holds 8-byte entries");

// The scratch itself: about 9 MB for kNoAllocMaxPairs = 2^20.
static __device__ __align__(256) uint32_t g_sort_scratch[kNoAllocWords];

constexpr int kNoAllocMaxDevices = 64;
struct NoAllocDevice {
  uint32_t* base = nullptr;  // device address of g_sort_scratch on this device
  SortWorkspace ws{};
};
std::mutex g_noalloc_mu;
NoAllocDevice g_noalloc[kNoAllocMaxDevices];

}  // namespace
}  // namespace gpulsm

extern "C" lsm_status lsm_sort_pairs_noalloc(const uint32_t* d_keys_in, const uint32_t* d_vals_in,
                                             uint32_t* d_keys_out, uint32_t* d_vals_out, uint64_t n,
                                             void* stream) {
  using namespace gpulsm;
  if (n > kNoAllocMaxPairs) return LSM_ERR_CAPACITY;
  if (n && (!d_keys_in || !d_vals_in || !d_keys_out || !d_vals_out)) return LSM_ERR_ARG;
  if (n == 0) return LSM_OK;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) {
    cudaGetLastError();
    return LSM_ERR_CUDA;
  }
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  NoAllocDevice& d = g_noalloc[dev];
  if (!d.base) {
    // Once per device, with that device current: the host needs the array's
    // device address (its name in host code is only a host-side stand-in),
    // and the control words must start at zero.
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_sort_scratch) != cudaSuccess || !p) {
      cudaGetLastError();
      return LSM_ERR_CUDA;
    }
    uint32_t* base = static_cast<uint32_t*>(p);
    if (cudaMemsetAsync(base, 0, kNoAllocCtl * sizeof(uint32_t), st) != cudaSuccess) {
      cudaGetLastError();
      return LSM_ERR_CUDA;
    }
    d.ws.ctl = base;
    d.ws.lookback = nullptr;
    d.ws.max_tiles = 0;
    d.ws.epoch = 0;
    d.ws.flip = 0;
    d.ws.sticky = base + kNoAllocSticky;
    d.ws.tilecnt = base + kNoAllocRuns;
    d.base = base;
  }
  SortArgs a{};
  a.mode = kSortPairs;
  a.in_keys = d_keys_in;
  a.in_vals = d_vals_in;
  a.n_in = n;
  a.n = uint32_t(n);
  a.out_keys = d_keys_out;
  a.out_vals = d_vals_out;
  a.tmp_keys = d.base + kNoAllocTmpK;
  a.tmp_vals = d.base + kNoAllocTmpV;
  // Each sort leaves the control block of the next one zeroed; the run table
  // and the tile scratch are fully rewritten by every call before they are
  // read, so nothing else needs zeroing.
  cudaError_t e = sort_launch(a, d.ws, st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return LSM_ERR_CUDA;
  }
  return LSM_OK;
}
