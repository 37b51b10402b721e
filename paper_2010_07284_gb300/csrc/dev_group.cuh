// Fused evaluation of a group of pointwise and N operators on one tile.
//
// A group is a sub-DAG of threshold atoms, not/and/or and N (Sec. 2) whose
// inputs are image channels or masks materialised by earlier steps.  Every
// value lives in a shared-memory buffer of (th + 2*halo) rows: the core tile
// plus `halo` rows above and below and one vector of four 32-px words left and
// right (of which the word next to the core counts).  A node whose value is needed `h` pixels beyond the core
// is computed over rows [halo - h, halo + th + h); N consumes one pixel of
// halo, so a chain of k N operators inside a group needs halo >= k (the
// compiler caps it at 31, inside the one-word horizontal margin).  Pixels
// outside the image are stored as 0 where a neighbour may read them, which is
// exactly the clipping of the neighbourhood at the image border.
#pragma once
#include "dev_common.cuh"

namespace vl {

// Mask slot k of a job.
VL_DEV uint32_t* slot_ptr(const DevJob& J, int k) {
  const size_t words = (size_t)J.H * J.Wp;
  if (k < J.n_inter_slots) return J.slot_mem + k * words;
  if (k < J.n_inter_slots + J.n_root_slots) return J.root_mem + (k - J.n_inter_slots) * words;
  return J.slots[k];
}

VL_DEV uint4 lds4(const uint32_t* p) { return *reinterpret_cast<const uint4*>(p); }
VL_DEV void sts4(uint32_t* p, uint4 v) { *reinterpret_cast<uint4*>(p) = v; }

// Barrier over the first n threads of the block (whole warps).
VL_DEV void group_sync(int n) { asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory"); }

// One tile of a group, as its threads see it.
//
// Buffers are rows of nv vectors of four words: the core tile's words (tiles
// have whole vectors of them), and a
// vector left and right of them (only the word next to the core
// matters: a halo is at most 31 pixels), so that every vector of a buffer
// starts at a 16-byte boundary of the mask it comes from.  Vector v of every
// buffer belongs to thread v mod EXEC_THREADS, for every instruction except
// the float threshold, so the compiler needs a block barrier (I_SYNC) only
// where a thread touches a word another thread touched since the last one.
struct GroupGeom {
  int r0, w0, th, tww;  // core tile: image row, image word, rows, words
  int halo, rows, nv;   // rows above and below it; rows and vectors of a buffer
  int vecs;             // vectors from one buffer to the next
};
VL_DEV GroupGeom group_geom(const DevJob& J, const StepDesc& S, int sub) {
  GroupGeom g;
  const int ty = sub / J.g_tiles_x, tx = sub - ty * J.g_tiles_x;
  g.r0 = ty * J.gth;
  g.w0 = tx * J.gtww;
  g.th = min(J.gth, J.H - g.r0);
  g.tww = min(J.gtww, J.Wp - g.w0);
  g.halo = S.halo;
  g.rows = g.th + 2 * S.halo;
  g.nv = group_vecs(J.gtww);
  g.vecs = (J.gth + 2 * S.halo) * g.nv;
  return g;
}

// Vector v of the buffers: it lies in the image's words whole or not at all.
struct GroupVec {
  int at;        // first word in a buffer
  int off;       // first word in a mask of the image
  int need;      // halo from which it is computed; huge: no such vector
  int row;       // the same for its row as a whole
  int hi;        // its pixels [0, hi) lie in the image (none: hi <= 0)
  int where;     // bit 0: first of its row, bit 1: last
  bool core;     // its words are the core tile's
  VL_DEV bool in() const { return hi > 0; }
  // the pixels of word k that lie in the image
  VL_DEV uint32_t mask(int k) const {
    const int n = hi - 32 * k;
    return n >= 32 ? 0xFFFFFFFFu : n <= 0 ? 0u : (1u << n) - 1u;
  }
  VL_DEV uint4 clip(uint4 v) const {
    if (hi == 128) return v;
    return make_uint4(v.x & mask(0), v.y & mask(1), v.z & mask(2), v.w & mask(3));
  }
};
VL_DEV GroupVec group_vec(const DevJob& J, const GroupGeom& g, int v) {
  GroupVec q;
  const int i = v / g.nv, jv = v - i * g.nv;
  q.at = 4 * v;
  // (the words left and right of the core are neighbours of something only
  // where there is a halo)
  q.where = (jv == 0 ? 1 : 0) | (jv == g.nv - 1 ? 2 : 0);
  q.row = i < g.rows ? max(g.halo - i, i - (g.halo + g.th - 1)) : 1 << 20;
  q.need = max(q.row, q.where ? 1 : 0);
  const int y = g.r0 - g.halo + i, wg = g.w0 - 4 + 4 * jv;
  q.hi = y >= 0 && y < J.H && wg >= 0 ? min(128, J.W - 32 * wg) : 0;
  q.off = y * J.Wp + wg;
  q.core = q.need <= 0 && 4 * (jv - 1) < g.tww;
  return q;
}
// Its words of the mask at g (0 outside the image), and back.
VL_DEV uint4 vec_load(const uint32_t* g, const GroupVec& q) {
  return q.in() ? __ldcg(reinterpret_cast<const uint4*>(g + q.off)) : make_uint4(0u, 0u, 0u, 0u);
}
VL_DEV void vec_store(uint32_t* g, const GroupVec& q, uint4 v) {
  if (q.core) *reinterpret_cast<uint4*>(g + q.off) = v;
}

// Instructions as the interpreter runs them, four words each:
//   x  offset of dst | offset of a << 16    (vectors from the first buffer)
//   y  offset of b | halo << 16 | P_PUT | P_* << 24 (and P_SYNC)
//   z, w  loads and stores: the mask's address; P_LOGIC: flips of a (and of
//      the result) and of b; P_NEAR: z connectivity; P_CONST: z the word;
//      P_RTHR: z the bound | code bits << 16 | lt << 31, w first word of the
//      staged planes (P_RTHR_FAR: first plane); P_THR: the channel plane's
//      address (56 bits) with TH_* above it, the bound's halves in place of
//      the operands' offsets
enum : uint32_t { P_END = 0, P_LOAD, P_STORE, P_LOGIC, P_NOT, P_NEAR, P_CONST, P_RTHR, P_RTHR_FAR,
                  P_THR };
constexpr uint32_t P_PUT = 1u << 23;   // the next instruction stores this value
constexpr uint32_t P_SYNC = 0x80u;     // with the opcode: a block barrier precedes
constexpr uint32_t TH_LT = 1u << 29, TH_U16 = 1u << 30, TH_WRITTEN = 1u << 31;

// A float threshold (a constant, or a percentile found earlier in the launch)
// into buffer d: the rows it is needed on, the tile's words that lie in the
// image, and the one left and right of them if a neighbour will be read (h >
// 0); further words lie outside the image, and nothing inside comes of them.
// A lane loads 4 pixels (16 bytes, or 8 of uint16), a warp 4 words a load and
// UNR loads in flight; three shuffles put four of them together.  By the whole
// block.  Not inlined: the interpreter's loop needs its registers.
//
// Bound by the latency of its loads: the groups of 1024 slices (six thresholds a
// pixel) take 877 us of the grid, and took 1157 with four loads in flight,
// twelve shuffles, a division a load, and words outside the image.
static __device__ __noinline__ void group_threshold(const DevJob& J, const StepDesc& S, int sub,
                                                    uint4 I, uint32_t* d) {
  constexpr int UNR = 8;
  const GroupGeom g = group_geom(J, S, sub);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, part = lane & 7, quad = lane >> 3;
  const int H = J.H, W = J.W, Wp = J.Wp, pitch = J.pitch, h = (I.y >> 16) & 0x7F;
  const void* plane = reinterpret_cast<const void*>(
      (unsigned long long)I.z | (unsigned long long)(I.w & 0xFFFFFFu) << 32);
  const int fmt = I.w & TH_U16 ? PX_U16 : PX_F32;
  const bool nc = !(I.w & TH_WRITTEN), lt = I.w & TH_LT;
  const float t = __uint_as_float((I.x >> 16) << 16 | (I.y & 0xFFFFu));
  const int side = h > 0 ? 1 : 0;
  const int bw = g.tww + 2 * side;  // words worked on in a row
  const int n = (g.th + 2 * h) * bw, y0 = g.r0 - h, w0 = g.w0 - side;
  // idx / bw as a product (exact: idx * bw < 2^32)
  const unsigned inv = bw > 1 ? 0xFFFFFFFFu / (unsigned)bw + 1u : 0u;
  auto row_of = [&](int idx) { return bw > 1 ? (int)__umulhi((unsigned)idx, inv) : idx; };
  d += (g.halo - h) * g.nv * 4 + 4 - side;
  for (int base = warp * 4 * UNR; base < n; base += EXEC_WARPS * 4 * UNR) {
    float4 v[UNR];
#pragma unroll
    for (int u = 0; u < UNR; ++u) {
      const int idx = base + 4 * u + quad, i = row_of(idx), wg = w0 + idx - i * bw, y = y0 + i;
      v[u] = idx < n && y >= 0 && y < H && wg >= 0 && wg < Wp
                 ? ld_px4(plane, fmt, nc, (size_t)y * pitch + 32 * wg + 4 * part)
                 : make_float4(t, t, t, t);  // (passes neither test)
    }
#pragma unroll
    for (int u0 = 0; u0 < UNR; u0 += 4) {
      uint32_t nib[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 x = v[u0 + u];
        nib[u] = lt ? ((x.x < t) | ((x.y < t) << 1) | ((x.z < t) << 2) | ((x.w < t) << 3))
                    : ((x.x > t) | ((x.y > t) << 1) | ((x.z > t) << 2) | ((x.w > t) << 3));
      }
      const uint32_t word = join_nibbles4(nib, part);
      const int idx = base + 4 * (u0 + (part >> 1)) + quad, i = row_of(idx), j = idx - i * bw;
      if (!(part & 1) && idx < n)
        d[i * g.nv * 4 + j] = w0 + j >= 0 ? word & vmask(w0 + j, W) : 0u;
    }
  }
}

// Stage of rank planes: plane after plane, the rows the group's thresholds
// need, nv - 1 vectors a row -- the core's, and one that packs the word
// right of the core (word 0) and the word left of it (word 3).  Every thread
// copies what it reads itself, so its own wait is enough.
VL_DEV int stage_plane_words(const StepDesc& S, const GroupGeom& g) {
  return (g.th + 2 * S.rank_halo) * (g.nv - 1) * 4;
}
// Words of the planes of the tables below `upto`.
VL_DEV int stage_words(const DevJob& J, const StepDesc& S, const GroupGeom& g, int upto) {
  int n = 0;
  for (unsigned m = (unsigned)S.rank_mask; m; m &= m - 1) {
    const int t = __ffs(m) - 1;
    if (t >= upto) break;
    n += J.rtab[t].nbits + 1;
  }
  return n * stage_plane_words(S, g);
}
VL_DEV int stage_at(const StepDesc& S, const GroupGeom& g, const GroupVec& q) {
  const int v = q.at >> 2, i = v / g.nv, jv = v - i * g.nv;
  return ((i - (g.halo - S.rank_halo)) * (g.nv - 1) + (q.where ? g.nv - 2 : jv - 1)) * 4;
}
VL_DEV void stage_copy(const DevJob& J, const StepDesc& S, const GroupGeom& g, const GroupVec& q,
                       uint32_t* stage) {
  if (q.need > S.rank_halo || !q.in()) return;
  const size_t pstride = (size_t)J.H * J.Wp;
  const int per_plane = stage_plane_words(S, g);
  uint32_t* dst = stage + stage_at(S, g, q);
  for (unsigned m = (unsigned)S.rank_mask; m; m &= m - 1) {
    const RankTab T = J.rtab[__ffs(m) - 1];
    const uint32_t* src = J.planes + (size_t)T.plane0 * pstride + q.off;
    for (int p = 0; p <= T.nbits; ++p, dst += per_plane, src += pstride) {
      if (q.where & 1) {
        if (q.mask(3)) cp_async4(dst + 3, src + 3);
      } else if (q.where) {
        if (q.mask(0)) cp_async4(dst, src);
      } else {
        cp_async16(dst, src);
      }
    }
  }
}

// code < K, bit-sliced: the subtraction code - K must borrow.  Bit b passes
// the borrow on as ~x_b | borrow where K_b = 1 and as ~x_b & borrow where
// K_b = 0, i.e. the majority of (~x_b, borrow, K_b) -- one logic op per
// plane.  Below K's lowest set bit no borrow starts, so the chain begins
// there (K = 0: never).
VL_DEV void rank_pass(uint4& w, uint4 x, uint32_t km) {
  w.x = (~x.x & w.x) | (~x.x & km) | (w.x & km);
  w.y = (~x.y & w.y) | (~x.y & km) | (w.y & km);
  w.z = (~x.z & w.z) | (~x.z & km) | (w.z & km);
  w.w = (~x.w & w.w) | (~x.w & km) | (w.w & km);
}
VL_DEV uint4 rank_result(uint4 w, uint4 nan, bool lt) {
  const uint32_t f = lt ? 0u : 0xFFFFFFFFu;
  return make_uint4((w.x ^ f) & ~nan.x, (w.y ^ f) & ~nan.y, (w.z ^ f) & ~nan.z, (w.w ^ f) & ~nan.w);
}

// The value of instruction I (no load, store or float threshold) on vector q.
// stage: the thread's place in the staged planes.
VL_DEV uint4 group_value(const DevJob& J, uint4 I, uint32_t op, const uint32_t* buf,
                         const GroupVec& q, int row_words, const uint32_t* stage, int per_plane) {
  const uint32_t* const a = buf + (I.x >> 16) * 4 + q.at;
  if (op == P_LOGIC) {
    const uint4 v = lds4(a), w = lds4(buf + (I.y & 0xFFFFu) * 4 + q.at);
    return make_uint4(((v.x ^ I.z) & (w.x ^ I.w)) ^ I.z, ((v.y ^ I.z) & (w.y ^ I.w)) ^ I.z,
                      ((v.z ^ I.z) & (w.z ^ I.w)) ^ I.z, ((v.w ^ I.z) & (w.w ^ I.w)) ^ I.z);
  }
  uint4 z;
  if (op == P_NEAR) {
    // rows above and below lie in the buffer: the operand is computed one
    // row further out.  Left of the first and right of the last vector
    // nothing is known; that is 128 pixels from the core.
    const int r = row_words;
    const uint4 u = lds4(a - r), m = lds4(a), n = lds4(a + r);
    uint32_t l = 0, e = 0;
    if (!(q.where & 1)) l = I.z == 8 ? a[-r - 1] | a[-1] | a[r - 1] : a[-1];
    if (!(q.where & 2)) e = I.z == 8 ? a[-r + 4] | a[4] | a[r + 4] : a[4];
    const uint4 o = make_uint4(u.x | n.x, u.y | n.y, u.z | n.z, u.w | n.w);
    const uint32_t f = I.z == 8 ? 0xFFFFFFFFu : 0u;
    z = near_vec(make_uint4(m.x | (o.x & f), m.y | (o.y & f), m.z | (o.z & f), m.w | (o.w & f)), o,
                 l, e);
  } else if (op == P_NOT) {
    const uint4 v = lds4(a);
    z = make_uint4(~v.x, ~v.y, ~v.z, ~v.w);
  } else if (op == P_CONST) {
    z = make_uint4(I.z, I.z, I.z, I.z);
  } else {
    uint4 w = make_uint4(0u, 0u, 0u, 0u), nan = w;
    const int nb = (I.z >> 16) & 0xFF;
    const uint32_t K = I.z & 0xFFFFu;
    const bool lt = I.z >> 31;
    const int b0 = K ? __ffs(K) - 1 : nb;
    if (op == P_RTHR) {
      const uint32_t* s0 = stage + I.w;
#pragma unroll 4
      for (int b = b0; b < nb; ++b) rank_pass(w, lds4(s0 + b * per_plane), 0u - ((K >> b) & 1u));
      if (lt) nan = lds4(s0 + nb * per_plane);
    } else {
      const size_t pstride = (size_t)J.H * J.Wp;
      const uint32_t* g = J.planes + (size_t)I.w * pstride;
#pragma unroll 4
      for (int b = b0; b < nb; ++b)
        rank_pass(w, vec_load(g + (size_t)b * pstride, q), 0u - ((K >> b) & 1u));
      if (lt) nan = vec_load(g + (size_t)nb * pstride, q);
    }
    z = rank_result(w, nan, lt);
  }
  return q.clip(z);
}

VL_DEV uint32_t* insn_ptr(uint4 I) {
  return reinterpret_cast<uint32_t*>((unsigned long long)I.z | ((unsigned long long)I.w << 32));
}

// Translates instructions [s0, s0 + cnt) of the group into prog, and an end
// mark; the first n_act threads.  (Read one by one while the group runs,
// instructions and the addresses of masks cost 500 cycles each.)
VL_DEV void group_translate(const DevJob& J, const StepDesc& S, const GroupGeom& g, int s0, int cnt,
                            int n_act, bool staged, uint32_t* prog) {
  const uint4* src = reinterpret_cast<const uint4*>(J.insns + S.insn_off + s0);
  for (int k = threadIdx.x; k <= cnt; k += n_act) {
    uint4 w = make_uint4(0u, P_END << 24, 0u, 0u);
    if (k < cnt) {
      const uint4 i = __ldg(src + k);
      const uint32_t op = i.x & 0x7Fu, dst = (i.x >> 8) & 0xFFu, a = (i.x >> 16) & 0xFFu, b = i.x >> 24;
      uint32_t p = P_LOGIC;
      w.x = dst * g.vecs | (a * g.vecs) << 16;
      w.y = b * g.vecs;
      if (op == I_LOAD || op == I_STORE) {
        p = op == I_LOAD ? P_LOAD : P_STORE;
        const unsigned long long m = (unsigned long long)slot_ptr(J, (int16_t)(i.y >> 16));
        w.z = (uint32_t)m;
        w.w = (uint32_t)(m >> 32);
      } else if (op == I_OR) {
        w.z = w.w = 0xFFFFFFFFu;
      } else if (op == I_ANDNOT) {
        w.w = 0xFFFFFFFFu;
      } else if (op == I_NOT) {
        p = P_NOT;
      } else if (op == I_NEAR) {
        p = P_NEAR;
        w.z = J.conn;
      } else if (op == I_CONST) {
        p = P_CONST;
        w.y = 0;
        w.z = b ? 0xFFFFFFFFu : 0u;
      } else if (op == I_RTHR) {
        p = staged ? P_RTHR : P_RTHR_FAR;
        w.x = dst * g.vecs;
        w.y = 0;
        w.z = (i.z & 0xFFFFu) | (i.z >> 16) << 16 | (b & 1u) << 31;
        w.w = staged ? (uint32_t)stage_words(J, S, g, (int)a) : i.y >> 16;
      } else if (op == I_THR) {
        p = P_THR;
        const DevImage im = J.images[(int16_t)i.z];
        const int slot = (int16_t)(i.y >> 16);
        const uint32_t t = slot >= 0 ? __float_as_uint(ldcg(J.pct_val + slot)) : i.w;
        const unsigned long long m = (unsigned long long)chan_ptr(im, (int)i.z >> 16, (size_t)J.H * J.pitch);
        w.x = dst * g.vecs | (t >> 16) << 16;
        w.y = t & 0xFFFFu;
        w.z = (uint32_t)m;
        w.w = ((uint32_t)(m >> 32) & 0xFFFFFFu) | ((b & 1u) ? TH_LT : 0u) |
              (im.format == PX_U16 ? TH_U16 : 0u) | (im.written ? TH_WRITTEN : 0u);
      }
      w.y |= (i.y & 0x7Fu) << 16;
      if (i.x & I_SYNC) p |= P_SYNC;
      if (p != P_STORE && p != P_THR && k + 1 < cnt) {
        const uint32_t n = __ldg(&src[k + 1].x);
        if ((n & 0xFFu) == I_STORE && ((n >> 16) & 0xFFu) == dst) w.y |= P_PUT;
      }
      w.y |= p << 24;
    }
    sts4(prog + 4 * k, w);
  }
}

// Masks of the loads ahead, fetched into a ring in shared memory, each vector
// by the thread that will use it: DEPTH (a power of two) entries of `entry`
// words.
struct GroupRing {
  uint32_t* base;            // the thread's vector of entry 0
  const uint16_t* load_at;   // which instructions are loads, 0xFFFF behind the last
  int entry;
};
template <int DEPTH>
VL_DEV void ring_fetch(const GroupRing& r, const uint32_t* prog, const GroupVec& q, int j) {
  const int k = r.load_at[j];
  if (k != 0xFFFF) {
    const uint4 w = lds4(prog + 4 * k);
    if (q.need <= (int)((w.y >> 16) & 0x7Fu) && q.in())
      cp_async16(r.base + (j & (DEPTH - 1)) * r.entry, insn_ptr(w) + q.off);
  }
  cp_async_commit();
}

// Runs a translated segment for a thread that owns one vector.  What bounds
// it is the chain through one instruction after the other, a few hundred
// cycles each for four to seven warps of a 14 x 32-word tile: so the loop
// keeps everything it needs in registers (spilled ones came back from L2,
// and cost more than the work), loads are fetched ahead, and a store behind
// the instruction that computes its value is done with it.
// Returns where it stopped: at the end, or at a float threshold, which the
// caller sees to (a call inside the loop would cost it registers).
template <int DEPTH>
VL_DEV const uint32_t* group_run(const DevJob& J, const uint32_t* prog, const uint32_t* pc, int& load,
                                 uint32_t* buf, const GroupVec& own, const GroupRing& ring,
                                 int row_words, const uint32_t* stage, int per_plane, int n_act) {
  uint4 next = lds4(pc);
  for (;;) {
    const uint4 I = next;
    const uint32_t op = (I.y >> 24) & 0x7Fu;
    if (op == P_END) return pc;
    if (I.y >> 31) group_sync(n_act);  // uniform: one instruction stream per CTA
    if (op == P_THR) return pc;
    pc += 4;
    next = lds4(pc);
    if (op == P_STORE) {
      if (own.core) vec_store(insn_ptr(I), own, lds4(buf + (I.x >> 16) * 4 + own.at));
      continue;
    }
    const bool mine = own.need <= (int)((I.y >> 16) & 0x7Fu);
    uint4 z = make_uint4(0u, 0u, 0u, 0u);
    if (op == P_LOAD) {
      if (DEPTH) {
        cp_async_wait<DEPTH ? DEPTH - 1 : 0>();  // the oldest fetch has landed
        if (mine && own.in()) z = lds4(ring.base + (load & (DEPTH - 1)) * ring.entry);
      } else if (mine) {
        z = vec_load(insn_ptr(I), own);
      }
    } else if (op == P_NEAR) {
      // the words beside the vector come from the lanes that hold the vectors
      // beside it (read from shared memory, at a stride of four words, they
      // took longer than the vectors); only the first and the last lane of a
      // warp read them.  All vectors of a row take part: the ones left and
      // right of the core are neighbours even where they need no value.
      const bool row = own.row <= (int)((I.y >> 16) & 0x7Fu);
      const uint32_t* const a = buf + (I.x >> 16) * 4 + own.at;
      const uint32_t f = I.z == 8 ? 0xFFFFFFFFu : 0u;
      uint4 o = make_uint4(0u, 0u, 0u, 0u), x = o;
      if (row) {
        const uint4 u = lds4(a - row_words), n = lds4(a + row_words);
        x = lds4(a);
        o = make_uint4(u.x | n.x, u.y | n.y, u.z | n.z, u.w | n.w);
        x = make_uint4(x.x | (o.x & f), x.y | (o.y & f), x.z | (o.z & f), x.w | (o.w & f));
      }
      uint32_t l = __shfl_up_sync(0xFFFFFFFFu, x.w, 1), e = __shfl_down_sync(0xFFFFFFFFu, x.x, 1);
      const int lane = threadIdx.x & 31;
      if (mine && lane == 0) l = a[-1] | ((a[-row_words - 1] | a[row_words - 1]) & f);
      if (mine && lane == 31) e = a[4] | ((a[-row_words + 4] | a[row_words + 4]) & f);
      if (own.where & 1) l = 0;
      if (own.where & 2) e = 0;
      z = own.clip(near_vec(x, o, l, e));
    } else if (mine) {
      if (op == P_RTHR) cp_async_wait<DEPTH>();  // the staged planes have landed
      z = group_value(J, I, op, buf, own, row_words, stage, per_plane);
    }
    if (mine) sts4(buf + (I.x & 0xFFFFu) * 4 + own.at, z);
    if (I.y & P_PUT) {
      if (own.core) vec_store(insn_ptr(next), own, z);
      pc += 4;
      next = lds4(pc);
    }
    if (DEPTH && op == P_LOAD) ring_fetch<DEPTH>(ring, prog, own, DEPTH + load++);
  }
}

// The same for a tile with more vectors than threads (one of many words, see
// tile_run_shape).
static __device__ __noinline__ void group_run_any(const DevJob& J, const StepDesc& S, int sub,
                                                  const uint32_t* prog, uint32_t* buf,
                                                  const uint32_t* stage) {
  const GroupGeom g = group_geom(J, S, sub);
  const int n = g.rows * g.nv, per_plane = stage_plane_words(S, g);
  cp_async_wait<0>();  // the staged planes have landed
  for (;; prog += 4) {
    const uint4 I = lds4(prog);
    const uint32_t op = (I.y >> 24) & 0x7Fu;
    if (op == P_END) break;
    if (I.y >> 31) group_sync(EXEC_THREADS);
    uint32_t* const d = buf + (I.x & 0xFFFFu) * 4;
    if (op == P_THR) {
      group_threshold(J, S, sub, I, d);
      continue;
    }
    for (int v = threadIdx.x; v < n; v += EXEC_THREADS) {
      const GroupVec q = group_vec(J, g, v);
      if (op == P_STORE) {
        vec_store(insn_ptr(I), q, lds4(buf + (I.x >> 16) * 4 + q.at));
      } else if (q.need <= (int)((I.y >> 16) & 0x7Fu)) {
        sts4(d + q.at, op == P_LOAD ? vec_load(insn_ptr(I), q)
                                    : group_value(J, I, op, buf, q, g.nv * 4,
                                                         stage + stage_at(S, g, q), per_plane));
      }
    }
  }
}

// A tile of a group.  smem: smem_words words of shared memory; buffers: most
// buffers a group of the plan may use.  Launched with EXEC_THREADS threads.
VL_DEV void group_tile(const DevJob& J, const StepDesc& S, int sub, uint32_t* smem, int smem_words,
                       int buffers) {
  constexpr int DEPTH = 4;
  const int tid = threadIdx.x, lane = tid & 31, n_insn = S.insn_cnt;
  const GroupGeom g = group_geom(J, S, sub);
  const bool one = g.rows * g.nv <= EXEC_THREADS;
  // threads that take part (a float threshold takes all); the others leave
  const int n_act = one && S.pct_cnt == 0 ? (g.rows * g.nv + 31) & ~31 : EXEC_THREADS;
  if (tid >= n_act) return;
  uint32_t* const prog = smem;
  uint32_t* const buf = smem + GROUP_PROG_BYTES / 4;
  uint32_t* rest = buf + min(max(S.n_bufs, 1), buffers) * g.vecs * 4;
  int room = smem_words - (int)(rest - smem);
  const GroupVec own = group_vec(J, g, tid);
  // the planes of the group's rank tables, when they fit
  const int st_words = stage_words(J, S, g, 32);
  const bool staged = S.rank_mask && st_words <= room;
  const uint32_t* stage = rest;
  if (staged) {
    if (one) {
      stage_copy(J, S, g, own, rest);
      stage += stage_at(S, g, own);
    } else {
      for (int v = tid; v < g.rows * g.nv; v += EXEC_THREADS)
        stage_copy(J, S, g, group_vec(J, g, v), rest);
    }
    rest += st_words;
    room -= st_words;
  }
  cp_async_commit();
  uint16_t* const load_at = reinterpret_cast<uint16_t*>(prog + 4 * (GROUP_SEG + 1));
  const GroupRing ring{rest + own.at, load_at, g.rows * g.nv * 4};
  const bool ahead = one && S.pct_off > 0 && room >= DEPTH * ring.entry;
  for (int s0 = 0; s0 < n_insn; s0 += GROUP_SEG) {
    const int cnt = min(GROUP_SEG, n_insn - s0);
    if (s0) group_sync(n_act);  // the segment before is done with its instructions
    group_translate(J, S, g, s0, cnt, n_act, staged, prog);
    group_sync(n_act);
    if (!one) {
      group_run_any(J, S, sub, prog, buf, stage);
      continue;
    }
    if (ahead) {
      if (tid < 32) {  // where the loads are
        int n = 0;
        for (int k = 0; k < cnt; k += 32) {
          const bool is = k + lane < cnt && ((prog[4 * (k + lane) + 1] >> 24) & 0x7Fu) == P_LOAD;
          const unsigned m = __ballot_sync(0xFFFFFFFFu, is);
          if (is) load_at[n + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(k + lane);
          n += __popc(m);
        }
        if (lane < DEPTH) load_at[n + lane] = 0xFFFF;
      }
      group_sync(n_act);
      for (int j = 0; j < DEPTH; ++j) ring_fetch<DEPTH>(ring, prog, own, j);
    }
    int load = 0;
    const uint32_t* pc = prog;
    for (;;) {
      const int per_plane = stage_plane_words(S, g);
      pc = ahead ? group_run<DEPTH>(J, prog, pc, load, buf, own, ring, g.nv * 4, stage, per_plane, n_act)
                 : group_run<0>(J, prog, pc, load, buf, own, ring, g.nv * 4, stage, per_plane, n_act);
      const uint4 I = lds4(pc);
      if (((I.y >> 24) & 0x7Fu) == P_END) break;
      group_threshold(J, S, sub, I, buf + (I.x & 0xFFFFu) * 4);
      pc += 4;
    }
  }
  cp_async_wait<0>();  // no copy may outlive the tile
}

}  // namespace vl
