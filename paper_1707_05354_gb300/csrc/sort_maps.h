// Key arithmetic of the batch sort: which bucket and sub-bin a key variable
// falls in, and which keys a round over a crowded bucket takes.  Plain integer
// functions without CUDA constructs, so that they can be checked on the host.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define GPULSM_HD __host__ __device__ __forceinline__
#else
#define GPULSM_HD inline
#endif

namespace gpulsm {

GPULSM_HD uint32_t mul_hi(uint32_t a, uint32_t b) { return uint32_t((uint64_t(a) * b) >> 32); }
GPULSM_HD uint32_t lesser(uint32_t a, uint32_t b) { return a < b ? a : b; }
GPULSM_HD uint32_t greater(uint32_t a, uint32_t b) { return a < b ? b : a; }
// a / b; the device's quotient may be off by a few units in the last place.
GPULSM_HD float quotient(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fdividef(a, b);
#else
  return a / b;
#endif
}
// The same rounded down to a whole number (from 2^32 on: 2^32 - 1).
GPULSM_HD uint32_t floor_quotient(float a, float b) {
#ifdef __CUDA_ARCH__
  return __float2uint_rd(quotient(a, b));
#else
  const float q = quotient(a, b);
  return q >= 4294967296.0f ? 0xFFFFFFFFu : uint32_t(q);
#endif
}

// The buckets of one sort: `parts` equal parts of the key range, part(kv) =
// floor((kv - lo) * mul / 2^32), and, of every hot key variable, a bucket of its
// own, which splits the part that holds it in two: in key order.
struct KeyMap {
  uint32_t lo, mul, parts, nhot;
  const uint32_t* hot;  // ascending
  GPULSM_HD uint32_t part(uint32_t kv) const { return lesser(mul_hi(greater(kv, lo) - lo, mul), parts - 1); }
  GPULSM_HD uint32_t bucket(uint32_t kv) const {
    uint32_t d = part(kv);
    for (uint32_t h = 0; h < nhot; ++h) d += (kv >= hot[h] ? 1u : 0u) + (kv > hot[h] ? 1u : 0u);
    return d;
  }
  // smallest key variable of part p in 1 .. parts - 1 (2^32 - 1 for a part the
  // 32 bits do not reach: key variables are below it)
  GPULSM_HD uint32_t lower(uint32_t p) const {
    const uint64_t kv = lo + ((uint64_t(p) << 32) + mul - 1) / mul;
    return kv < 0xFFFFFFFFull ? uint32_t(kv) : 0xFFFFFFFFu;
  }
  // `parts` parts of the range [lo, hi] that 512 samples span, widened by 1/50
  // at both ends: evenly spread keys reach beyond it with a probability of
  // about e^-10 at either end, 512 / 50.  (What does falls in the first or last
  // sub-bin; more than a few there and the bucket takes 8-bit passes.  With
  // 1/128, e^-4, that was one batch in fifty at either end: four rounds of 34
  // batches of 30000 took 256 us, now 244; one sort of 2^20 24.9 and 25.0.)
  static GPULSM_HD KeyMap spanning(uint32_t lo, uint32_t hi, uint32_t parts, uint32_t nhot, const uint32_t* hot) {
    const uint32_t ext = (hi - lo) / 50 + 1;
    const uint32_t l = lo > ext ? lo - ext : 0u, h = hi < ~ext ? hi + ext : 0xFFFFFFFFu;
    // (a float quotient: any factor near parts * 2^32 / range does, the same in
    // every CTA)
    const uint32_t q = floor_quotient(float(parts) * 4294967296.0f, float(h - l) + 1.0f);
    return KeyMap{l, greater(1u, q), parts, nhot, hot};
  }
};

// Few equal parts, 2^bits <= 256 of them: runs of the parts of a map of 256.
// (The factor of a map of two parts over nearly 2^32 keys is 2 or 3, whole, so
// that one of them could get two thirds of the range and overflow: four rounds
// of 128 batches of 8192 keys below 2^30 took 435 us, now 252.)
struct PartMap {
  KeyMap fine;
  uint32_t drop;
  static GPULSM_HD PartMap of(uint32_t lo, uint32_t mul, uint32_t bits) {
    return PartMap{KeyMap{lo, mul, 256u, 0u, nullptr}, 8u - bits};
  }
  static GPULSM_HD PartMap spanning(uint32_t lo, uint32_t hi, uint32_t bits) {
    return PartMap{KeyMap::spanning(lo, hi, 256u, 0u, nullptr), 8u - bits};
  }
  GPULSM_HD uint32_t part(uint32_t kv) const { return fine.part(kv) >> drop; }
  GPULSM_HD uint32_t lower(uint32_t p) const { return fine.lower(p << drop); }
  // about the key variables of a part
  static GPULSM_HD float width(uint32_t mul, uint32_t bits) {
    return quotient(1099511627776.0f, float(mul) * float(1u << bits)) + 1.0f;
  }
};

// Sub-bin of kv: floor((kv - off) * mul / 2^32), for kv below base as for
// base, kept below kSubBins; monotone.
constexpr uint32_t kSubBins = 4096;  // counting pass over a bucket's elements
struct SubMap {
  uint32_t base, off, mul;
  // `width` key variables from base: for up to kSubBins of them each has a
  // sub-bin of its own (off = base - 1: (x + 1) (2^32 - 1) / 2^32 is x)
  static GPULSM_HD SubMap of(uint32_t base, float width) {
    if (width <= float(kSubBins)) return SubMap{base, base - 1u, 0xFFFFFFFFu};
    return SubMap{base, base, floor_quotient(float(1ull << 44), width)};
  }
  GPULSM_HD uint32_t sub(uint32_t kv) const { return lesser(mul_hi(greater(kv, base) - off, mul), kSubBins - 1); }
  // the largest key variable of sub-bin s
  GPULSM_HD uint32_t last(uint32_t s) const {
    return off + uint32_t(((uint64_t(s + 1) << 32) + mul - 1) / mul) - 1;
  }
};
static_assert(kSubBins == 4096, "2^44 = kSubBins * 2^32");

// The keys [a, b] that the rounds over a crowded bucket have still to do: at
// first all keys there are, whatever range the bucket is said to have, so that
// every element has its turn and the rounds end.
struct KeyTurn {
  uint32_t a = 0u, b = 0xFFFFFFFFu;
  // The next round takes the elements' range [mn, mx] in sub-bins and looks at
  // the first `fit` of them (at least one; fewer than reach mx).
  GPULSM_HD void narrow(uint32_t mn, const SubMap& map, uint32_t fit) {
    a = mn;
    b = map.last(fit ? fit - 1 : 0u);
  }
  // [a, b] is done.
  GPULSM_HD void next() {
    a = b + 1;
    b = 0xFFFFFFFFu;
  }
};

}  // namespace gpulsm
