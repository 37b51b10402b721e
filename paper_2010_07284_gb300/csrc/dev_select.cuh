// Exact order statistic of one image channel: the percentile of level q is
// the value of rank floor(q*(n-1)) in ascending order, no interpolation (the
// "percentiles" normalisation of Sec. 4.2).  Keys are order-preserving
// integers: a float's bits (NaN sorts after +infinity), or a uint16 pixel.
//
// A sample of the channel gives two keys that most likely enclose the wanted
// one and few others.  One pass over the channel counts what lies below,
// at and between them; what lies between (some percent of the channel) is
// then taken apart by histograms of 12 bits of its range at a time.  A count
// that shows the rank outside, or at one of the two keys (a background value
// that many pixels share), needs no second guess: the range is then what is
// left on that side, or the key itself.
//
// (All of it is inlined where shared memory is known by name, and channels go
// by value: behind pointers, atomics would be generic ones and a channel's
// fields would be read again after every store.)
//
// Two forms.  One block per select (select_rank), for batches of selects that
// fill the GPU: the keys between go to a list in shared memory, unless they
// are too many for it.  Many blocks per select (sel_pass, sel_range), for a
// few selects on large channels: counts and histograms are added up in global
// memory, and every block works out the range found so far from them, so that
// no pass of its own does.
//
// What bounds a select is instructions and the loads in front of them: a
// block alone on its SM reads 3 pixels a ns, and has about 10 us of sample,
// sort and histograms of its list to do besides.  Five selects of the four
// float channels of a 155 x 240 x 240 scan over the whole grid: 60 us for the
// pass that counts (70 with the ends of the range counted behind a branch),
// 34 us (5.2 TB/s, partly from L2) for the one after it.  The three passes of one block per select
// that histogrammed every pixel's digits before took 1.82 ms for three
// 1021 x 1530 channels where this takes 35 us, and 124 us for a 240 x 240 one
// (two blocks on an SM) where this takes 40; bound by atomics on shared
// memory, that form read 0.8 pixels a ns in whatever way its bins were laid
// out.
#pragma once
#include "dev_common.cuh"
#include "select_range.h"

namespace vl {

VL_DEV float sel_float(uint32_t key) { return __uint_as_float(sel_key_bits(key)); }

constexpr int SEL_SAMPLE = 1024;
struct SelectSmem {
  uint32_t hist[SEL_BINS];            // (the sample, while it is sorted)
  uint32_t part[EXEC_WARPS];
  uint32_t digit, below;              // bin holding the rank, keys below it
  uint32_t count[4];                  // keys below, at the lower, at the upper key, between
};
static_assert(SEL_SAMPLE == 2 * EXEC_THREADS, "a thread sorts two keys");

// A channel: rows of `pitch` elements, W of them pixels.
struct SelChan {
  const void* p;
  int format, nc, H, W, pitch;
  VL_DEV unsigned vpr() const { return (unsigned)(W + 3) >> 2; }
  VL_DEV unsigned vecs() const { return (unsigned)H * vpr(); }
  VL_DEV uint32_t top() const { return format == PX_U16 ? 0xFFFFu : 0xFFFFFFFFu; }
  VL_DEV float value(uint32_t key) const { return format == PX_U16 ? (float)key : sel_float(key); }
};

// f(keys) for all pixels of vectors [v0, v1) of the channel (a vector: four
// pixels of a row; pitches are multiples of 128 elements), SEL_KEYS at a time,
// by the whole block; whole warps call f together.  Where there is no pixel a
// key is the highest one: such keys come after all pixels' in any order, and
// no rank reaches them.  Row and column are stepped, not divided out.
constexpr int SEL_UNR = 4, SEL_KEYS = 4 * SEL_UNR;
template <bool U16, class F>
VL_DEV void sel_scan_t(SelChan c, unsigned v0, unsigned v1, F f) {
  const unsigned nt = blockDim.x, vpr = c.vpr();
  const unsigned sy = nt / vpr, sx = nt - sy * vpr;
  unsigned i = v0 + threadIdx.x, y = i / vpr, x = i - y * vpr;
  for (unsigned base = v0 + (threadIdx.x & ~31u); base < v1; base += SEL_UNR * nt) {
    uint4 raw[SEL_UNR];
    const uint32_t top = U16 ? 0xFFFFFFFFu : SEL_TOP_BITS;
#pragma unroll
    for (int u = 0; u < SEL_UNR; ++u) {
      raw[u] = make_uint4(top, top, top, top);
      if (i < v1) {
        const size_t at = (size_t)y * c.pitch + 4 * x;
        const int n = c.W - (int)(4 * x);
        if (U16) {
          const uint2 w = __ldg(reinterpret_cast<const uint2*>(static_cast<const unsigned short*>(c.p) + at));
          raw[u].x = w.x;
          raw[u].y = w.y;
          if (n < 4) {
            raw[u].x |= n < 2 ? 0xFFFF0000u : 0u;
            raw[u].y |= n < 3 ? 0xFFFFFFFFu : 0xFFFF0000u;
          }
        } else {
          const uint4* w = reinterpret_cast<const uint4*>(static_cast<const float*>(c.p) + at);
          raw[u] = c.nc ? __ldg(w) : __ldcg(w);
          if (n < 4) {
            raw[u].w = top;
            if (n < 3) raw[u].z = top;
            if (n < 2) raw[u].y = top;
          }
        }
      }
      i += nt;
      y += sy;
      x += sx;
      if (x >= vpr) { x -= vpr; ++y; }
    }
    uint32_t k[SEL_KEYS];
#pragma unroll
    for (int u = 0; u < SEL_UNR; ++u) {
      if (U16) {
        k[4 * u] = raw[u].x & 0xFFFFu;
        k[4 * u + 1] = raw[u].x >> 16;
        k[4 * u + 2] = raw[u].y & 0xFFFFu;
        k[4 * u + 3] = raw[u].y >> 16;
      } else {
        k[4 * u] = sel_key(raw[u].x);
        k[4 * u + 1] = sel_key(raw[u].y);
        k[4 * u + 2] = sel_key(raw[u].z);
        k[4 * u + 3] = sel_key(raw[u].w);
      }
    }
    f(k);
  }
}
template <class F>
VL_DEV void sel_scan(SelChan c, unsigned v0, unsigned v1, F f) {
  if (c.format == PX_U16) sel_scan_t<true>(c, v0, v1, f);
  else sel_scan_t<false>(c, v0, v1, f);
}

// Finds the bin of h[0 .. SEL_BINS) that holds `rank` (s.digit) and the keys
// below it (s.below).  h: shared memory, or global memory written by other
// blocks.  A block barrier before (for h in shared memory) and at the end.
VL_DEV void sel_pick(SelectSmem& s, const uint32_t* h, bool global, unsigned long long rank) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int PER = SEL_BINS / EXEC_THREADS;
  static_assert(PER == 8, "two vectors");
  const uint4* h4 = reinterpret_cast<const uint4*>(h) + 2 * tid;
  const uint4 u = global ? __ldcg(h4) : h4[0], v = global ? __ldcg(h4 + 1) : h4[1];
  const uint32_t b[PER] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
  uint32_t sum = 0;
#pragma unroll
  for (int q = 0; q < PER; ++q) sum += b[q];
  uint32_t incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) s.part[warp] = incl;
  __syncthreads();
  uint32_t before = 0;  // of the warps before
#pragma unroll
  for (int w = 0; w < EXEC_WARPS; ++w) before += w < warp ? s.part[w] : 0u;
  unsigned long long acc = (unsigned long long)before + incl - sum;
  if (sum > 0 && acc <= rank && rank < acc + sum) {  // exactly one thread
    int q = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j)
      if (q == j && acc + b[j] <= rank) {
        acc += b[j];
        q = j + 1;
      }
    s.digit = (uint32_t)(tid * PER + q);
    s.below = (uint32_t)acc;
  }
  __syncthreads();
}

// Two keys that most likely enclose the key of rank k: order statistics of a
// sample, 3.5 standard deviations of its rank to either side; the ends of the
// key range where the sample ends, or where it would not be worth its sort.
// One key of every 1/SEL_SAMPLE of the channel, at a place that a
// multiplicative hash gives (evenly spaced ones would all lie in one column
// of many images).  By the whole block; a block barrier at the end.
VL_DEV SelRange sel_sample(SelectSmem& s, SelChan c, long long k) {
  SelRange r{0u, c.top(), 0ull};
  const long long n = (long long)c.H * c.W;
  if (n <= 4 * SEL_SAMPLE) return r;
  const unsigned long long nv = c.vecs();
  const unsigned vpr = c.vpr();
  uint32_t* key = s.hist;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const unsigned j = threadIdx.x + h * EXEC_THREADS, u = j * 0x9E3779B1u;
    const unsigned v = (unsigned)((j * nv + ((u * nv) >> 32)) / SEL_SAMPLE);
    const unsigned y = v / vpr, x = v - y * vpr, px = 4 * x + ((u >> 12) & 3u);
    const size_t at = (size_t)y * c.pitch + min(px, (unsigned)c.W - 1u);
    if (c.format == PX_U16) key[j] = __ldg(static_cast<const unsigned short*>(c.p) + at);
    else key[j] = sel_key(c.nc ? __ldg(static_cast<const uint32_t*>(c.p) + at)
                               : __ldcg(static_cast<const uint32_t*>(c.p) + at));
  }
  __syncthreads();
  for (unsigned size = 2; size <= SEL_SAMPLE; size *= 2)  // bitonic sort
    for (unsigned step = size / 2; step > 0; step /= 2) {
      // (steps up to 32 stay within the 64 keys of a warp)
      if (step >= 32) __syncthreads();
      else __syncwarp();
      const unsigned i = 2 * threadIdx.x - (threadIdx.x & (step - 1)), j = i + step;
      const uint32_t a = key[i], b = key[j];
      if ((a > b) == ((i & size) == 0)) {
        key[i] = b;
        key[j] = a;
      }
    }
  __syncthreads();
  const float q = (float)k / (float)n, at = q * SEL_SAMPLE;
  const float dev = 3.5f * sqrtf(SEL_SAMPLE * q * (1.f - q)) + 2.f;
  const int a = (int)floorf(at - dev), b = (int)ceilf(at + dev);
  if (a >= 0) r.lo = key[min(a, SEL_SAMPLE - 1)];
  if (b < SEL_SAMPLE) r.hi = key[max(b, 0)];
  __syncthreads();
  return r;
}

// Counts of the sample's keys over vectors [v0, v1) into s.count, and
// between(keys, which) for the keys between them (whole warps).  (Keys at r.lo
// are not counted at r.hi again where the two are the same.)
template <class F>
VL_DEV void sel_count(SelectSmem& s, SelChan c, const SelRange& r, unsigned v0, unsigned v1,
                      F between) {
  uint32_t lt = 0, at_lo = 0, at_hi = 0, in = 0;
  // key - lo: below it wraps around, 0 and span are the ends, and one less is
  // below span - 1 between them
  const uint32_t span = r.hi - r.lo, inner = span ? span - 1u : 0u;
  sel_scan(c, v0, v1, [&](const uint32_t (&k)[SEL_KEYS]) {
    uint32_t m = 0;
#pragma unroll
    for (int q = 0; q < SEL_KEYS; ++q) {
      const uint32_t d = k[q] - r.lo;
      lt += k[q] < r.lo;
      at_lo += d == 0;
      at_hi += d == span;
      if (d - 1u < inner) m |= 1u << q;
    }
    in += __popc(m);
    between(k, m);
  });
  if (r.lo == r.hi) at_hi = 0;
  lt = __reduce_add_sync(0xFFFFFFFFu, lt);
  at_lo = __reduce_add_sync(0xFFFFFFFFu, at_lo);
  at_hi = __reduce_add_sync(0xFFFFFFFFu, at_hi);
  in = __reduce_add_sync(0xFFFFFFFFu, in);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&s.count[0], lt);
    atomicAdd(&s.count[1], at_lo);
    atomicAdd(&s.count[2], at_hi);
    atomicAdd(&s.count[3], in);
  }
}

VL_DEV void sel_clear(SelectSmem& s) {
  for (int i = threadIdx.x; i < SEL_BINS; i += blockDim.x) s.hist[i] = 0;
}

// One block selects rank k of the channel.  list: room for `cap` keys in
// shared memory.  Returns the value in every thread (after a block barrier).
VL_DEV float select_rank(SelectSmem& s, uint32_t* list, int cap, SelChan c, long long k,
                         int32_t* status) {
  const unsigned n = c.vecs();
  const int lane = threadIdx.x & 31;
  const SelRange guess = sel_sample(s, c, k);
  if (threadIdx.x < 4) s.count[threadIdx.x] = 0;
  if (threadIdx.x == 4) s.digit = 0;  // (keys listed)
  __syncthreads();
  sel_count(s, c, guess, 0, n, [&](const uint32_t (&key)[SEL_KEYS], uint32_t m) {
    const int mine = __popc(m);
    int at = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xFFFFFFFFu, at, o);
      if (lane >= o) at += t;
    }
    const int all = __shfl_sync(0xFFFFFFFFu, at, 31);
    if (all == 0) return;
    int first = 0;
    if (lane == 0) first = (int)atomicAdd(&s.digit, (uint32_t)all);
    at += __shfl_sync(0xFFFFFFFFu, first, 0) - mine;
#pragma unroll
    for (int q = 0; q < SEL_KEYS; ++q)
      if ((m >> q) & 1u) {
        if (at < cap) list[at] = key[q];
        ++at;
      }
  });
  __syncthreads();
  bool between;
  SelRange r = sel_resolve(guess, c.top(), s.count, k, between);
  const uint32_t listed = s.count[3];
  const bool from_list = between && listed <= (uint32_t)cap;
  for (int round = 0; round < SEL_ROUNDS && !r.done(); ++round) {
    sel_clear(s);
    __syncthreads();
    if (from_list) {
      for (unsigned i = threadIdx.x; i < listed; i += blockDim.x)
        if (r.holds(list[i])) atomicAdd(&s.hist[r.bin(list[i])], 1u);
    } else {
      sel_scan(c, 0, n, [&](const uint32_t (&key)[SEL_KEYS]) {
#pragma unroll
        for (int q = 0; q < SEL_KEYS; ++q)
          if (r.holds(key[q])) atomicAdd(&s.hist[r.bin(key[q])], 1u);
      });
    }
    __syncthreads();
    sel_pick(s, s.hist, false, r.rank);
    r.take(s.digit, s.below);
  }
  if (!r.done() && threadIdx.x == 0) set_status(status, ST_INTERNAL | RS_SELECT);
  __syncthreads();
  return c.value(r.lo);
}

// A select over many blocks, in global memory (SEL_HIST words, zeroed): the
// sample's keys, the four counts, then a histogram per pass.
struct SelShared {
  uint32_t lo, hi, count[4];
  uint32_t key, done;  // the key, once a block found it (written together)
  uint32_t pad[8];
};
VL_DEV uint32_t* sel_hist_of(uint32_t* g, int pass) {
  return g + sizeof(SelShared) / 4 + pass * SEL_BINS;
}

// The range that `passes` finished passes leave (one at least).
VL_DEV SelRange sel_range(SelectSmem& s, uint32_t* g, SelChan c, int passes, long long k) {
  const uint4 a = __ldcg(reinterpret_cast<const uint4*>(g));
  const uint2 b = __ldcg(reinterpret_cast<const uint2*>(g + 4)), e = __ldcg(reinterpret_cast<const uint2*>(g + 6));
  // (every thread has to see the same: the block that writes it may be ahead)
  if (__syncthreads_or((int)e.y)) {
    const uint32_t key = __ldcg(g + 6);
    return SelRange{key, key, 0ull};
  }
  const uint32_t count[4] = {a.z, a.w, b.x, b.y};
  bool between;
  SelRange r = sel_resolve(SelRange{a.x, a.y, 0ull}, c.top(), count, k, between);
  for (int p = between ? 0 : 1; p < passes && !r.done(); ++p) {
    sel_pick(s, sel_hist_of(g, p), true, r.rank);
    r.take(s.digit, s.below);
  }
  return r;
}

// Block `block` of `blocks` of pass `pass`: its share of the channel.
VL_DEV void sel_pass(SelectSmem& s, SelChan c, int pass, int block,
                                             int blocks, long long k, uint32_t* g) {
  const unsigned n = c.vecs(), per = (n + blocks - 1) / blocks;
  const unsigned v0 = min(n, block * per), v1 = min(n, v0 + per);
  if (pass == 0) {
    const SelRange guess = sel_sample(s, c, k);
    const SelRange in{guess.lo + 1u, guess.hi - 1u, 0ull};
    sel_clear(s);
    if (threadIdx.x < 4) s.count[threadIdx.x] = 0;
    __syncthreads();
    sel_count(s, c, guess, v0, v1, [&](const uint32_t (&key)[SEL_KEYS], uint32_t m) {
#pragma unroll
      for (int q = 0; q < SEL_KEYS; ++q)
        if ((m >> q) & 1u) atomicAdd(&s.hist[in.bin(key[q])], 1u);
    });
    __syncthreads();
    if (threadIdx.x < 4 && s.count[threadIdx.x]) atomicAdd(g + 2 + threadIdx.x, s.count[threadIdx.x]);
    if (threadIdx.x == 4) g[0] = guess.lo;  // (every block writes the same)
    if (threadIdx.x == 5) g[1] = guess.hi;
  } else {
    const SelRange r = sel_range(s, g, c, pass, k);
    if (r.done()) {
      if (block == 0 && threadIdx.x == 0) *reinterpret_cast<uint2*>(g + 6) = make_uint2(r.lo, 1u);
      return;
    }
    sel_clear(s);
    __syncthreads();
    sel_scan(c, v0, v1, [&](const uint32_t (&key)[SEL_KEYS]) {
#pragma unroll
      for (int q = 0; q < SEL_KEYS; ++q)
        if (r.holds(key[q])) atomicAdd(&s.hist[r.bin(key[q])], 1u);
    });
    __syncthreads();
  }
  uint32_t* out = sel_hist_of(g, pass);
  for (int i = threadIdx.x; i < SEL_BINS; i += blockDim.x)
    if (s.hist[i]) atomicAdd(out + i, s.hist[i]);
}

// The value of rank k from finished passes.
VL_DEV float sel_finish(SelectSmem& s, uint32_t* g, SelChan c, long long k) {
  return c.value(sel_range(s, g, c, SEL_PASSES, k).lo);
}

}  // namespace vl
