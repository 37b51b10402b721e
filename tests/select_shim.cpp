// Test shim: a percentile select over the range arithmetic of
// paper_2010_07284_gb300/csrc/select_range.h, compiled with the host compiler
// by tests/test_select_range.py.
#include <vector>

#include "select_range.h"

extern "C" unsigned sel_key_of(unsigned bits) { return vl::sel_key(bits); }
extern "C" unsigned sel_bits_of(unsigned key) { return vl::sel_key_bits(key); }

// Key of rank k among n keys, starting from the guess [lo, hi].  Returns the
// number of histograms it took, or -1: more than `limit` of them, a bin out of
// range, or a histogram without the rank.
extern "C" int sel_run(const unsigned* key, int n, long long k, unsigned lo, unsigned hi, unsigned top,
                       int limit, unsigned* out) {
  uint32_t count[4] = {0, 0, 0, 0};
  for (int i = 0; i < n; ++i) {
    if (key[i] < lo) ++count[0];
    else if (key[i] == lo) ++count[1];
    else if (key[i] < hi) ++count[3];
    else if (key[i] == hi) ++count[2];
  }
  bool between;
  vl::SelRange r = vl::sel_resolve(vl::SelRange{lo, hi, 0ull}, top, count, k, between);
  int rounds = 0;
  for (; !r.done(); ++rounds) {
    if (rounds == limit) return -1;
    std::vector<uint32_t> h(4096, 0);
    for (int i = 0; i < n; ++i)
      if (r.holds(key[i])) {
        if (r.bin(key[i]) >= h.size()) return -1;
        ++h[r.bin(key[i])];
      }
    uint32_t digit = 0, below = 0;
    while (digit < h.size() && below + h[digit] <= r.rank) below += h[digit++];
    if (digit == h.size()) return -1;
    r.take(digit, below);
  }
  *out = r.lo;
  return rounds;
}
