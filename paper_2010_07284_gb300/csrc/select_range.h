// Integer arithmetic of the percentile selects (dev_select.cuh), also compiled
// for the host: order-preserving keys of float bits, and ranges of keys that
// are narrowed by histograms of 12 bits of the range at a time.
#pragma once
#include <stdint.h>

#include "vl_internal.h"

namespace vl {

VL_HD_INLINE int sel_clz(uint32_t x) {
#if defined(__CUDA_ARCH__)
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}

// Key of a float's bits: ordered like the float, -infinity at 0 and every NaN
// above +infinity (the negative ones, whose bits sort below -infinity, wrap
// around to the top).
VL_HD_INLINE uint32_t sel_key(uint32_t u) {
  return (u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u)) - 0x007FFFFFu;
}
VL_HD_INLINE uint32_t sel_key_bits(uint32_t key) {
  const uint32_t k = key + 0x007FFFFFu;
  return (k & 0x80000000u) ? k ^ 0x80000000u : ~k;
}
constexpr uint32_t SEL_TOP_BITS = 0xFF800001u;  // the float bits of the highest key

// Histograms that take any range down to one key: 12 bits each of 32, so that
// 20, 8 and no bits of the distance of its ends are left.
constexpr int SEL_ROUNDS = 3;

// Keys [lo, hi] among which the wanted one has rank `rank`.
struct SelRange {
  uint32_t lo, hi;
  unsigned long long rank;
  VL_HD_INLINE bool done() const { return lo == hi; }
  // bits of key - lo below a bin
  VL_HD_INLINE int shift() const {
    const int sh = 20 - sel_clz(hi - lo);
    return sh > 0 ? sh : 0;
  }
  VL_HD_INLINE uint32_t bin(uint32_t key) const { return (key - lo) >> shift(); }
  VL_HD_INLINE bool holds(uint32_t key) const { return key - lo <= hi - lo; }
  // The range of bin `digit`, with `below` keys in the bins below it.  Its end
  // is found as a distance: as a key it may lie past 2^32 (a range that ends
  // at the highest keys has a last bin that reaches beyond them).
  VL_HD_INLINE void take(uint32_t digit, uint32_t below) {
    const int sh = shift();
    const uint32_t last = (1u << sh) - 1u;
    lo += digit << sh;
    if (hi - lo > last) hi = lo + last;
    rank -= below;
  }
};

// The range that the counts below, at and between the sample's keys leave for
// rank k of the channel.  `between`: it is the one between them.
VL_HD_INLINE SelRange sel_resolve(const SelRange& r, uint32_t top, const uint32_t* count, long long k,
                                  bool& between) {
  unsigned long long rank = (unsigned long long)k;
  between = false;
  if (rank < count[0]) return SelRange{0u, r.lo - 1u, rank};
  rank -= count[0];
  if (rank < count[1]) return SelRange{r.lo, r.lo, rank};
  rank -= count[1];
  between = rank < count[3];
  if (between) return SelRange{r.lo + 1u, r.hi - 1u, rank};
  rank -= count[3];
  if (rank < count[2]) return SelRange{r.hi, r.hi, rank};
  return SelRange{r.hi + 1u, top, rank - count[2]};
}

}  // namespace vl
