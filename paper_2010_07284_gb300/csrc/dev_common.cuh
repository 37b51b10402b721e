// Small device helpers shared by every kernel of the library.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "vl_internal.h"

#define VL_DEV __device__ __forceinline__

namespace vl {

// Bits of word w (of a row of width W) that are real pixels.
VL_DEV uint32_t vmask(int w, int W) {
  int n = W - 32 * w;
  return n >= 32 ? 0xFFFFFFFFu : (n <= 0 ? 0u : ((1u << n) - 1u));
}

// Mask of bits 0..b inclusive.
VL_DEV uint32_t le_mask(int b) { return b >= 31 ? 0xFFFFFFFFu : ((2u << b) - 1u); }

// Row and column of element i of a row-major grid of `cols` columns: a
// 32-bit division while i < 2^32 (every word index, and every pixel index
// of a grid under 2^32 pixels), else a 64-bit one.
VL_DEV void split_index(long long i, int cols, int& row, int& col) {
  if (i < (1LL << 32)) {
    const unsigned u = (unsigned)i, c = (unsigned)cols, r = u / c;
    row = (int)r;
    col = (int)(u - r * c);
  } else {
    row = (int)(i / cols);
    col = (int)(i - (long long)row * cols);
  }
}

// Loads that bypass L1: data written by other CTAs of the same launch.
VL_DEV uint32_t ldcg(const uint32_t* p) { return __ldcg(p); }
VL_DEV int32_t ldcg(const int32_t* p) { return __ldcg(p); }
VL_DEV float ldcg(const float* p) { return __ldcg(p); }
VL_DEV uint8_t ldcg(const uint8_t* p) {
  return (uint8_t)__ldcg((const unsigned char*)p);
}

// Asynchronous copies to shared memory, in groups per thread.
VL_DEV void cp_async4(uint32_t* smem_dst, const uint32_t* gmem_src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gmem_src) : "memory");
}
VL_DEV void cp_async16(uint32_t* smem_dst, const uint32_t* gmem_src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}
VL_DEV void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// Waits until at most N of this thread's latest copy groups are unfinished.
template <int N>
VL_DEV void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// First error wins.
VL_DEV void set_status(int32_t* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

// Horizontal dilation of word c given its left/right neighbour words.
VL_DEV uint32_t hdil(uint32_t l, uint32_t c, uint32_t r) {
  return c | (c << 1) | (l >> 31) | (c >> 1) | (r << 31);
}

// Dilated word from a 3x3 neighbourhood of words (rows u, m, d; columns
// left, centre, right).  conn 8: square; conn 4: cross.
VL_DEV uint32_t near_word(uint32_t ul, uint32_t uc, uint32_t ur, uint32_t ml,
                          uint32_t mc, uint32_t mr, uint32_t dl, uint32_t dc,
                          uint32_t dr, int conn) {
  if (conn == 8) return hdil(ul, uc, ur) | hdil(ml, mc, mr) | hdil(dl, dc, dr);
  return uc | dc | hdil(ml, mc, mr);
}

// N on a vector of four words x, given the words left and right of it in the
// row: for the square, of the three rows around together (o = x); for the
// cross, of its own row, with o the rows above and below.
VL_DEV uint4 near_vec(uint4 x, uint4 o, uint32_t l, uint32_t e) {
  return make_uint4(o.x | hdil(l, x.x, x.y), o.y | hdil(x.x, x.y, x.z), o.z | hdil(x.y, x.z, x.w),
                    o.w | hdil(x.z, x.w, e));
}
VL_DEV uint4 or4(uint4 a, uint4 b) { return make_uint4(a.x | b.x, a.y | b.y, a.z | b.z, a.w | b.w); }
// Vector jv of a row without the bits that are no pixels.
VL_DEV uint4 clip_vec(uint4 v, int jv, int W) {
  if (128 * (jv + 1) <= W) return v;
  return make_uint4(v.x & vmask(4 * jv, W), v.y & vmask(4 * jv + 1, W), v.z & vmask(4 * jv + 2, W),
                    v.w & vmask(4 * jv + 3, W));
}

// The 8 lanes of a group hold the nibbles n[u] of four 32-pixel words u (lane
// `sub` pixels 4 * sub ..): returns word sub >> 1.  Three shuffles: half of
// the words change sides with the other four lanes, then one of two with the
// lane two further, then the halves of a word are joined.
VL_DEV uint32_t join_nibbles4(const uint32_t (&n)[4], int sub) {
  const int h = 4 * (sub & 3);
  const uint32_t x = (n[0] | n[1] << 16) << h, y = (n[2] | n[3] << 16) << h;
  const bool high = sub & 4, second = sub & 2;
  const uint32_t own = high ? y : x, other = __shfl_xor_sync(0xFFFFFFFFu, high ? x : y, 4);
  const uint32_t lo = high ? other : own, hi = high ? own : other;
  const uint32_t w0 = __byte_perm(lo, hi, 0x5410), w1 = __byte_perm(lo, hi, 0x7632);
  uint32_t w = second ? w1 : w0;
  w |= __shfl_xor_sync(0xFFFFFFFFu, second ? w0 : w1, 2);
  return w | __shfl_xor_sync(0xFFFFFFFFu, w, 1);
}

// ---- number images: float or uint16 planes of H x pitch elements
// (a uint16 pixel is its integer value, exact in float)

// Channel ch of image im; plane_elems = H * pitch.
VL_DEV const void* chan_ptr(const DevImage& im, int ch, size_t plane_elems) {
  const size_t esz = im.format == PX_U16 ? 2 : 4;
  return static_cast<const char*>(im.data) + (size_t)ch * plane_elems * esz;
}

// Element i of a channel plane.  `nc`: the read-only path may be used (the
// image is not written during the launch).
VL_DEV float ld_px(const void* p, int format, bool nc, size_t i) {
  if (format == PX_U16) return (float)__ldg(static_cast<const unsigned short*>(p) + i);
  const float* f = static_cast<const float*>(p) + i;
  return nc ? __ldg(f) : __ldcg(f);
}

// Elements i .. i+3 (i a multiple of 4: 16- or 8-byte aligned).
VL_DEV float4 ld_px4(const void* p, int format, bool nc, size_t i) {
  if (format == PX_U16) {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(static_cast<const unsigned short*>(p) + i));
    return make_float4((float)(u.x & 0xFFFFu), (float)(u.x >> 16), (float)(u.y & 0xFFFFu),
                       (float)(u.y >> 16));
  }
  const float4* f = reinterpret_cast<const float4*>(static_cast<const float*>(p) + i);
  return nc ? __ldg(f) : __ldcg(f);
}

}  // namespace vl
