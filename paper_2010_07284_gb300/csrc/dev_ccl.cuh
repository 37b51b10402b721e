// Connected components on bit-packed masks, and the component select that
// reachability reduces to (Sec. 3.2: rho phi1[phi2] = N(phi1 or Z), Z the
// phi2-components that meet N phi1).
//
// Design (sm_103a, union-find, no host round trips -- unlike the paper's
// iterated pointer jumping with host-checked termination, Sec. 3.3):
//   1. tile-local: one CTA labels a tile of CCL_TH rows x CCL_TWW words.
//      The union-find elements are the connected pieces of two-row strips,
//      found with bit operations on the packed words; they are united in
//      shared memory with atomicMin, over all strip boundaries at once.
//   2. publish: every foreground pixel on the tile border, and every local
//      root that reaches the border, gets an entry G[gid] in a global
//      union-find array indexed by linear pixel id gid = y*W + x.
//   3. merge: pixels adjacent across tile borders are united in G; a root
//      is linked under the smaller root by compare-and-swap, so only a node
//      that is still a root is ever re-pointed and links always point to
//      smaller gids (no cycles).
//   4. final: each tile takes up what it saved, resolves its border roots in
//      G, and writes labels or the selected components.
// Labels are canonical: the minimum linear index of each component.
#pragma once
#include <climits>

#include "dev_common.cuh"

namespace vl {

constexpr uint32_t FULL = 0xFFFFFFFFu;

// Pairs the first links of a tile may leave over (more are united at once).
constexpr int CCL_PEND = 4096;
static_assert(CCL_MAXRUNS <= 16384, "runs are packed into 16 bits with two flags");

struct CclSmem {
  static constexpr bool SEEDS = true;
  uint32_t m[CCL_TH][CCL_TWW];   // rows of the tile
  uint32_t u[CCL_NS][CCL_TWW];   // strip unions (row 2k | row 2k+1)
  uint32_t st[CCL_NS][CCL_TWW];  // strip-run starts
  uint32_t sd[CCL_NS][CCL_TWW];  // first seed column of every strip run, per word
  int32_t pre[CCL_NS][CCL_TWW];  // starts before each word, per strip
  int32_t qc[CCL_NS][CCL_TWW];   // boundary anchor entering each word
  int32_t cnt[CCL_NS];           // runs of each strip
  int32_t base[CCL_NS + 1];      // first strip-run id of each strip
  int32_t npend;                 // pairs offered to pend (may exceed its size)
  int32_t nlist;                 // border roots listed
  uint32_t pend[CCL_PEND];       // unions left over by the first links: run << 16 | run;
                                 //   later the list of border roots
  int32_t parent[CCL_MAXRUNS];   // union-find; after labelling a root holds -(value + 2)
  uint8_t flag[CCL_MAXRUNS];     // of roots: bit0 seed, bit1 on tile border
};

// What the select pass of rho keeps of a tile: its rows and strips, and a
// 16-bit code per strip run (the run's root, or for a root RZ_ROOT with
// RZ_SEED when it holds a seed pixel and RZ_SEL when it is selected).
constexpr uint32_t RZ_ROOT = 0x8000u, RZ_SEED = 0x4000u, RZ_SEL = 0x2000u;
struct RzSmem {
  static constexpr bool SEEDS = false;
  uint32_t m[CCL_TH][CCL_TWW];
  uint32_t u[CCL_NS][CCL_TWW];
  uint32_t st[CCL_NS][CCL_TWW];
  int32_t pre[CCL_NS][CCL_TWW];
  int32_t cnt[CCL_NS];
  int32_t base[CCL_NS + 1];
  uint32_t list[CCL_MAXBORDER];  // border roots: run | RZ_SEL << 16 when selected
  uint16_t code[CCL_MAXRUNS];
};

struct CclGeom {
  int H, W, Wp;
  int r0, w0;   // tile origin: image row, image word
  int th, tww;  // rows and words of this tile
};

// Tile `tile` of an image of H rows, or of a volume stored as its slices of
// Hs rows stacked (H = depth * Hs; Hs = H for an image): tiles never
// straddle two slices, so the tile-local labelling stays inside one slice.
// cth: rows of a tile (an even number up to CCL_TH; smaller tiles give small
// images more tiles to spread over the GPU).
VL_DEV CclGeom ccl_geom(int H, int W, int Wp, int tile, int tiles_x, int Hs, int cth = CCL_TH) {
  CclGeom g;
  g.H = H; g.W = W; g.Wp = Wp;
  const int tys = (Hs + cth - 1) / cth;  // tile rows per slice
  const int ty = tile / tiles_x, tx = tile - ty * tiles_x;
  const int z = ty / tys, tyz = ty - z * tys;
  g.r0 = z * Hs + tyz * cth;
  g.w0 = tx * CCL_TWW;
  g.th = min(cth, Hs - tyz * cth);
  g.tww = min(CCL_TWW, Wp - g.w0);
  return g;
}

VL_DEV int warp_incl_scan(int v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int t = __shfl_up_sync(FULL, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// ---------------------------------------------------------- shared u-f --

// cap = strip runs + 64: an index outside the runs, or a walk longer than
// cap, returns -1 (the caller reports RS_SUNION) instead of reading past
// the array.
VL_DEV int s_find(int32_t* par, int x, int cap) {
  volatile int32_t* p = par;
  if ((unsigned)x >= (unsigned)(cap - 64)) return -1;
  for (int it = 0; it < cap; ++it) {
    int q = p[x];
    if (q == x) return x;
    int r = p[q];
    if (r != q) p[x] = r;  // path halving: r is an ancestor of x
    x = q;
  }
  return -1;
}

// Roots of a and b, both chains walked side by side with path halving (each
// node passed is pointed at its grandparent, and the walk jumps there): on
// return a == b when the walks met (the same set; not necessarily a root),
// else both are roots.  False if an index is out of range or a bounded loop
// ran out (impossible unless memory is corrupted).
VL_DEV bool s_find2(int32_t* par, int& a, int& b, int cap) {
  volatile int32_t* p = par;
  const unsigned lim = (unsigned)(cap - 64);
  for (int it = 0; it < cap; ++it) {
    if (a == b) return true;
    if ((unsigned)a >= lim || (unsigned)b >= lim) return false;
    const int qa = p[a], qb = p[b];
    const bool ra = qa == a, rb = qb == b;
    if (ra && rb) return true;
    if ((unsigned)qa >= lim || (unsigned)qb >= lim) return false;
    const int ga = ra ? qa : p[qa], gb = rb ? qb : p[qb];
    if (!ra) {
      if (ga != qa) p[a] = ga;
      a = ga;
    }
    if (!rb) {
      if (gb != qb) p[b] = gb;
      b = gb;
    }
  }
  return false;
}

// Unite the sets of a and b; the smaller root wins.  Returns false if a
// bounded loop ran out (impossible unless memory is corrupted).
VL_DEV bool s_union(int32_t* par, int a, int b, int cap) {
  for (int it = 0; it < cap; ++it) {
    a = s_find(par, a, cap);
    b = s_find(par, b, cap);
    if (a < 0 || b < 0) return false;
    if (a == b) return true;
    if (a < b) { int t = a; a = b; b = t; }
    int old = atomicMin(&par[a], b);
    if (old == a) return true;
    a = old;
  }
  return false;
}

// ---------------------------------------------------------- global u-f --

// Root of x in G.  With `compress`, every node on the path from x gets the
// root as its parent.  This is safe because a node's parent only ever moves
// to one of its ancestors: g_union links a node only while it is a root
// (compare-and-swap), and nodes on the path from x, and the root found, all
// lie on x's single chain of ancestors, the root above them (ids decrease
// along the chain).  In the final labelling pass G is the label array and
// finished tiles have written their labels into it: the label of every
// node on a path is the root the path ends at, the value a compression
// writes there too.
// npx: entries of G.  An entry outside [0, npx) can only come from
// corrupted state; it is reported (reason RS_GRANGE) and the walk stops at
// the last valid node instead of reading out of bounds.
VL_DEV int g_find(int32_t* G, int x, int npx, int32_t* status, bool compress = true) {
  const int cap = min(npx + 64, 1 << 22);
  if ((unsigned)x >= (unsigned)npx) {
    set_status(status, ST_INTERNAL | RS_GRANGE);
    return 0;
  }
  int root = x;
  int it = 0;
  for (; it < cap; ++it) {
    const int p = ldcg(&G[root]);
    if (p == root) break;
    if ((unsigned)p >= (unsigned)npx) {
      set_status(status, ST_INTERNAL | RS_GRANGE);
      return root;
    }
    root = p;
  }
  if (it == cap) {
    set_status(status, ST_INTERNAL | RS_GFIND);
    return root;
  }
  if (compress) {
    for (int k = 0; k < it && x > root; ++k) {
      const int p = ldcg(&G[x]);
      if (p <= root) break;
      G[x] = root;
      x = p;
    }
  }
  return root;
}

// Roots of a and b in G, both chains walked side by side, with path halving:
// each node passed is pointed at its grandparent.  Like the compression in
// g_find this only ever moves a node to one of its ancestors, and it costs no
// second walk.  On return a == b (same set; they need not be roots) or both
// are roots.  Only while the union-find is being built: in the final pass a
// node of a finished tile holds its final label, which a halving write would
// replace by an inner node.
VL_DEV void g_find2(int32_t* G, int& a, int& b, int npx, int32_t* status) {
  const int cap = min(npx + 64, 1 << 22);
  for (int it = 0; it < cap; ++it) {
    if (a == b) return;
    if ((unsigned)a >= (unsigned)npx || (unsigned)b >= (unsigned)npx) {
      set_status(status, ST_INTERNAL | RS_GRANGE);
      a = b = 0;
      return;
    }
    const int pa = ldcg(&G[a]), pb = ldcg(&G[b]);
    const bool ra = pa == a, rb = pb == b;
    if (ra && rb) return;
    if ((unsigned)pa >= (unsigned)npx || (unsigned)pb >= (unsigned)npx) {
      set_status(status, ST_INTERNAL | RS_GRANGE);
      a = b = 0;
      return;
    }
    const int ga = ra ? pa : ldcg(&G[pa]), gb = rb ? pb : ldcg(&G[pb]);
    if (!ra) {
      if (ga != pa) G[a] = ga;
      a = ga;
    }
    if (!rb) {
      if (gb != pb) G[b] = gb;
      b = gb;
    }
  }
  set_status(status, ST_INTERNAL | RS_GFIND);
  a = b = 0;
}

// Unite the sets of a and b: the larger root is linked under the smaller,
// by compare-and-swap so that only a node that is still a root is ever
// re-pointed.  (An atomicMin on a root that was linked meanwhile would move
// its whole tree to the other set for a moment; a concurrent compression
// following that fresh link could then carry a node of the other set into
// this one and strand the rest of that set.)  A failed swap retries from
// fresh roots.
VL_DEV void g_union(int32_t* G, int a, int b, int npx, int32_t* status) {
  const int cap = min(npx + 64, 1 << 22);
  for (int it = 0; it < cap; ++it) {
    g_find2(G, a, b, npx, status);
    if (a == b) return;
    if (a < b) { int t = a; a = b; b = t; }
    if (atomicCAS(&G[a], a, b) == a) return;
  }
  set_status(status, ST_INTERNAL | RS_GUNION);
}

// ------------------------------------------------------- tile labelling --
//
// Level 0 is bit-parallel: in a strip of two rows A (top) and B, the
// components under 8-adjacency are exactly the runs of A | B (consecutive
// set columns always touch, diagonally at least); under 4-adjacency they are
// those runs cut where the set row switches from A-only to B-only (or back)
// between two columns.  These "strip runs" are the union-find elements.
// Strips are then merged across the CCL_NS - 1 strip boundaries.
// Across a boundary (rows A' = last row of the upper strip, B' = first row of
// the lower one), the same two-row rule holds: every set pixel of A' and B'
// inside one run of A' | B' (cut the same way for 4-adjacency) is connected,
// so each row run starting inside it is united with the run's anchor.

// The lowest bit of x in every segment of a 32-bit word, segments starting
// at bit 0 and at every set bit of s: clear the bits of x that have another
// bit of x below them in the same segment.  "Has an x bit below in its
// segment" is the carry into that position of P + x, P = ~s | x: a carry
// starts at every x bit, runs on through positions not in s, and dies at
// a bit of s that is not in x.
VL_DEV uint32_t first_in_segments(uint32_t x, uint32_t s) {
  const uint32_t p = ~s | x;
  const uint32_t carry_in = (p + x) ^ p ^ x;
  return x & ~(carry_in & ~s);
}

// Strip-run starts of a two-row strip (a, b) given the previous word's
// (a, b) (0 at the tile's left edge).
VL_DEV uint32_t strip_starts(uint32_t a, uint32_t b, uint32_t al, uint32_t bl, int conn) {
  const uint32_t u = a | b, ul = al | bl;
  uint32_t st = u & ~((u << 1) | (ul >> 31));
  if (conn == 4) {
    const uint32_t ao = a & ~b, bo = b & ~a, aol = al & ~bl, bol = bl & ~al;
    st |= (((ao << 1) | (aol >> 31)) & bo) | (((bo << 1) | (bol >> 31)) & ao);
  }
  return st;
}

// Strip run holding tile pixel x of strip k (x must be set in the strip).
template <class Smem>
VL_DEV int sid(const Smem& s, int k, int x) {
  const int w = x >> 5;
  return s.base[k] + s.pre[k][w] + __popc(s.st[k][w] & le_mask(x & 31)) - 1;
}

// Root of strip run i once roots are encoded (parent[root] < 0).
VL_DEV int root_of(const CclSmem& s, int i) {
  const int p = s.parent[i];
  return p >= 0 ? p : i;
}

// The two rows of the warp's strip (a warp takes one: a tile has no more
// strips than the block has warps), loaded ahead of ccl_tile_strips.
static_assert(EXEC_WARPS >= CCL_NS, "a warp per strip");
struct StripRows { uint32_t a, b; };
VL_DEV StripRows ccl_load_rows(const uint32_t* mask, const CclGeom& g) {
  const int lane = threadIdx.x & 31, r0 = 2 * (threadIdx.x >> 5);
  StripRows q{0u, 0u};
  if (lane < g.tww && r0 < g.th) {
    const size_t at = (size_t)(g.r0 + r0) * g.Wp + g.w0 + lane;
    q.a = ldcg(&mask[at]);
    if (r0 + 1 < g.th) q.b = ldcg(&mask[at + g.Wp]);
  }
  return q;
}

// Rows of the tile into shared memory, strip unions, strip-run starts, their
// counts before each word and per strip, and, with phi1, the seed columns (Smem::SEEDS):
// all loads of a strip are in flight together.  Every warp then adds the
// strips' counts up for itself: lane l returns the number of strip runs
// before strip l (lane 31: all of them), the same in every warp.  s.base is
// written by warp 0: a block barrier before it is read.
template <class Smem>
VL_DEV int ccl_tile_strips(Smem& s, StripRows rows, const uint32_t* phi1, const CclGeom& g, int conn) {
  const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
  const int ns = (g.th + 1) >> 1;
  if (k < ns) {
    const int y = g.r0 + 2 * k, w = g.w0 + lane;
    const bool in = lane < g.tww;
    uint32_t f[4] = {0u, 0u, 0u, 0u}, e[4] = {0u, 0u, 0u, 0u};
    if (phi1 != nullptr) {
      // phi1 around the strip, rows y - 1 .. y + 2 of the image, and beside
      // the tile, left of lane 0 and right of the last lane (a tile has at
      // least four words: they are two lanes)
      const int we = lane == 0 ? w - 1 : w + 1;
      const bool edge = in && (lane == 0 || lane == g.tww - 1) && we >= 0 && we < g.Wp;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int yy = y - 1 + q;
        const bool row = yy >= 0 && yy < g.H;
        if (row && in) f[q] = ldcg(&phi1[(size_t)yy * g.Wp + w]);
        if (row && edge) e[q] = ldcg(&phi1[(size_t)yy * g.Wp + we]);
      }
    }
    // padding bits (columns >= W) are cleared here, so that no later pass
    // can see a pixel outside the image whatever the caller's buffer holds
    const uint32_t vm = in ? vmask(w, g.W) : 0u, a = rows.a & vm, b = rows.b & vm;
    uint32_t al = __shfl_up_sync(FULL, a, 1), bl = __shfl_up_sync(FULL, b, 1);
    if (lane == 0) al = bl = 0;
    const uint32_t st = strip_starts(a, b, al, bl, conn);
    const int c = __popc(st);
    const int incl = warp_incl_scan(c, lane);
    s.m[2 * k][lane] = a;
    s.m[2 * k + 1][lane] = b;
    s.u[k][lane] = a | b;
    s.st[k][lane] = st;
    s.pre[k][lane] = incl - c;
    if (lane == 31) s.cnt[k] = incl;
    if (phi1 != nullptr) {
      // N phi1 on the two rows: vertical first, then the neighbour words
      uint32_t c0, c1, v0 = 0, v1 = 0, e0, e1;
      if (conn == 8) {
        c0 = f[0] | f[1] | f[2];
        c1 = f[1] | f[2] | f[3];
        e0 = e[0] | e[1] | e[2];
        e1 = e[1] | e[2] | e[3];
      } else {
        c0 = f[1];
        c1 = f[2];
        v0 = f[0] | f[2];
        v1 = f[1] | f[3];
        e0 = e[1];
        e1 = e[2];
      }
      uint32_t l0 = __shfl_up_sync(FULL, c0, 1), l1 = __shfl_up_sync(FULL, c1, 1);
      uint32_t q0 = __shfl_down_sync(FULL, c0, 1), q1 = __shfl_down_sync(FULL, c1, 1);
      if (lane == 0) { l0 = e0; l1 = e1; }
      if (lane == g.tww - 1) { q0 = e0; q1 = e1; }
      const uint32_t z = (a & (v0 | hdil(l0, c0, q0))) | (b & (v1 | hdil(l1, c1, q1)));
      if constexpr (Smem::SEEDS) s.sd[k][lane] = first_in_segments(z, st);
    }
  }
  __syncthreads();
  const int v = lane < ns ? s.cnt[lane] : 0;
  const int incl = warp_incl_scan(v, lane);
  if (k == 0) {
    if (lane < ns) s.base[lane] = incl - v;
    if (lane == 31) s.base[ns] = incl;
  }
  return lane == 31 ? incl : incl - v;
}

// Label one tile in shared memory.  Returns the number of strip runs, or -1
// (uniformly) if the tile has more than the shared arrays hold, which cannot
// happen for CCL_TH x CCL_TWW tiles; the caller then skips the tile.  On
// success: s.parent[i] of a non-root is its root (smallest id); a root holds
// a negative value -(v + 2).  With phi1 (the select of rho), v is a border
// pixel of the component (INT_MIN: it has none) and s.flag[root] bit0 says
// whether it holds a seed pixel (mask and N phi1); without (labels), v is
// the component's minimum linear pixel index.  s.pend[0 .. s.nlist) lists
// the roots of the components that reach the tile border.  Must be called by
// every thread of the block; a block barrier at the end.
VL_DEV int ccl_tile_label(CclSmem& s, const uint32_t* mask, const uint32_t* phi1,
                          const CclGeom& g, int conn, int32_t* status) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nw = blockDim.x >> 5;
  const int ns = (g.th + 1) >> 1;
  const int before = ccl_tile_strips(s, ccl_load_rows(mask, g), phi1, g, conn);
  const int nruns = __shfl_sync(FULL, before, 31);
  if (nruns > CCL_MAXRUNS) {  // uniform: every warp has the same count
    set_status(status, ST_INTERNAL | RS_TRUNS);
    return -1;
  }
  for (int i = tid; i < nruns; i += blockDim.x) {
    s.parent[i] = i;
    s.flag[i] = 0;
  }
  if (tid == 0) s.npend = s.nlist = 0;
  // 2. anchor of the boundary run entering each word from the left: the strip
  // run of its first pixel (in the upper strip if the upper row is set there)
  for (int b = warp; b < ns - 1; b += nw) {
    const int base_b = __shfl_sync(FULL, before, b), base_c = base_b + s.cnt[b];
    uint32_t A = 0, B = 0;
    if (lane < g.tww) { A = s.m[2 * b + 1][lane]; B = s.m[2 * b + 2][lane]; }
    uint32_t Al = __shfl_up_sync(FULL, A, 1), Bl = __shfl_up_sync(FULL, B, 1);
    if (lane == 0) Al = Bl = 0;
    const uint32_t qs = strip_starts(A, B, Al, Bl, conn);
    int last = -1;
    if (qs) {
      const int p = 31 - __clz(qs);
      last = (A >> p) & 1u ? base_b + s.pre[b][lane] + __popc(s.st[b][lane] & le_mask(p)) - 1
                           : base_c + s.pre[b + 1][lane] + __popc(s.st[b + 1][lane] & le_mask(p)) - 1;
    }
    int idx = last >= 0 ? lane : -1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, idx, o);
      if (lane >= o) idx = max(idx, t);
    }
    int prev = __shfl_up_sync(FULL, idx, 1);
    if (lane == 0) prev = -1;
    const int carried = __shfl_sync(FULL, last, prev < 0 ? 0 : prev);
    s.qc[b][lane] = prev < 0 ? -1 : carried;
  }
  __syncthreads();
  // 3. unite across the strip boundaries, all of them at once.  Every thread
  // takes a share of the columns of one boundary word; the word's strip data
  // sits in registers.  A row-run start ("event") links the larger of its
  // run and the boundary run's anchor under the smaller without looking for
  // roots: most runs (more than half of the events on noise) are linked
  // upwards for the first time and are done with that one atomicMin.  An
  // event whose run already had another parent leaves the pair (old parent,
  // smaller run) in a list, so that the parents and the list together always
  // hold the whole relation.
  const int cap = nruns + 64;
  bool ok = true;
  {
    const int pairs = (ns - 1) * g.tww;
    int T = 1;
    while (pairs > 0 && T < 32 && T * 2 * pairs <= (int)blockDim.x) T *= 2;
    const int pair = tid / T, sub = tid - pair * T;
    uint32_t A = 0, qs = 0, evA = 0, evB = 0, stb = 0, stc = 0;
    int bb = 0, bc = 0, carry = -1;
    if (pair < pairs) {
      const int b = pair / g.tww, w = pair - b * g.tww;
      A = s.m[2 * b + 1][w];
      const uint32_t B = s.m[2 * b + 2][w];
      const uint32_t Al = w > 0 ? s.m[2 * b + 1][w - 1] : 0u;
      const uint32_t Bl = w > 0 ? s.m[2 * b + 2][w - 1] : 0u;
      qs = strip_starts(A, B, Al, Bl, conn);
      stb = s.st[b][w];
      stc = s.st[b + 1][w];
      bb = s.base[b] + s.pre[b][w] - 1;
      bc = s.base[b + 1] + s.pre[b + 1][w] - 1;
      carry = s.qc[b][w];
      // one event per (boundary run, strip run): keep a row-run start only
      // when a boundary-run or strip-run start separates it from the
      // previous one, i.e. the first row-run start of every segment that
      // begins at such a start (or at the word's left edge)
      const uint32_t share = T == 1 ? FULL : (((1u << (32 / T)) - 1u) << (sub * (32 / T)));
      evA = first_in_segments(A & ~((A << 1) | (Al >> 31)), qs | stb) & share;
      evB = first_in_segments(B & ~((B << 1) | (Bl >> 31)), qs | stc) & share;
    }
    // links u and v; true when that left the pair (old, lo)
    auto link = [&](int u, int v, int& old, int& lo) {
      if (u == v) return false;
      const int hi = max(u, v);
      lo = min(u, v);
      old = atomicMin(&s.parent[hi], lo);
      return old != hi && old != lo;
    };
    auto push = [&](bool left, int old, int lo) {
      const unsigned lm = __ballot_sync(FULL, left);
      if (!lm) return;
      int at = 0;
      if (lane == 0) at = atomicAdd(&s.npend, __popc(lm));
      at = __shfl_sync(FULL, at, 0) + __popc(lm & ((1u << lane) - 1u));
      if (left) {
        if (at < CCL_PEND) s.pend[at] = ((uint32_t)old << 16) | (uint32_t)lo;
        else ok = s_union(s.parent, old, lo, cap) && ok;  // (the list is full)
      }
    };
    for (int round = 0; round < 32; ++round) {  // (at most 32 columns a word)
      const uint32_t ev = evA | evB;
      if (!__any_sync(FULL, ev != 0)) break;
      bool left1 = false, left2 = false;
      int old1 = 0, lo1 = 0, old2 = 0, lo2 = 0;
      if (ev) {
        const uint32_t bit = ev & (0u - ev), le = bit | (bit - 1u);
        const int ub = bb + __popc(stb & le), uc = bc + __popc(stc & le);
        const uint32_t qq = qs & le;
        int v = carry;
        if (qq) {
          const int q = 31 - __clz(qq);
          v = (A >> q) & 1u ? bb + __popc(stb & le_mask(q)) : bc + __popc(stc & le_mask(q));
        }
        if (v >= 0) {
          if (evA & bit) left1 = link(ub, v, old1, lo1);
          if (evB & bit) left2 = link(uc, v, old2, lo2);
        }
        evA &= ~bit;
        evB &= ~bit;
      }
      push(left1, old1, lo1);
      push(left2, old2, lo2);
    }
  }
  __syncthreads();
  // the listed pairs, dealt out evenly: both roots at once (walks that meet
  // need no link), the larger linked under the smaller; a link that finds
  // the larger root already linked elsewhere leaves the follow-up union
  // (old parent, smaller root) to the same thread
  {
    const int n = min(s.npend, CCL_PEND);
    int next = tid, pu = -1, pv = -1;
    for (int round = 0; round < 4 * CCL_MAXRUNS; ++round) {
      if (pu < 0 && next < n) {
        const uint32_t e = s.pend[next];
        pu = (int)(e >> 16);
        pv = (int)(e & 0xFFFFu);
        next += blockDim.x;
      }
      if (!__any_sync(FULL, pu >= 0)) break;
      if (pu >= 0) {
        int ra = pu, rb = pv;
        pu = -1;
        if (!s_find2(s.parent, ra, rb, cap)) {
          ok = false;
        } else if (ra != rb) {
          const int hi = max(ra, rb), lo = min(ra, rb);
          const int old = atomicMin(&s.parent[hi], lo);
          if (old != hi && old != lo) { pu = old; pv = lo; }
        }
      }
    }
  }
  __syncthreads();
  // 4. flatten: every thread points its own runs at their roots with finds
  // that only read, and marks its own roots INT_MIN.  (A path-halving find
  // writes grandparents into the entries it passes; landing after another
  // thread's final write to one of them, such a write would leave that run
  // one hop short of its root.)  Other threads' writes only move entries
  // closer to the roots, so a read-only walk still ends at the root.
  {
    volatile int32_t* vp = s.parent;
    for (int i = tid; i < nruns; i += blockDim.x) {
      int x = i, it = 0;
      for (; it < cap; ++it) {
        const int q = vp[x];
        if (q == x || q < 0) break;
        if ((unsigned)q >= (unsigned)nruns) { it = cap; break; }
        x = q;
      }
      if (it == cap) { ok = false; x = i; }
      vp[i] = x == i ? INT_MIN : x;
    }
  }
  if (!ok) set_status(status, ST_INTERNAL | RS_SUNION);
  __syncthreads();
  // 5. seeds: components holding a pixel of mask and N phi1
  if (phi1 != nullptr) {
    for (int k = warp; k < ns; k += nw) {
      uint32_t z = lane < g.tww ? s.sd[k][lane] : 0u;
      const uint32_t st = s.st[k][lane];
      const int id = s.base[k] + s.pre[k][lane] - 1;
      while (z) {
        const uint32_t bit = z & (0u - z);
        z ^= bit;
        s.flag[root_of(s, id + __popc(st & (bit | (bit - 1u))))] = 1;
      }
    }
    // (flags are bytes and the border marks below are word atomics)
    __syncthreads();
  }
  // 6. components on the tile border: the run starts of the first and the
  // last row, and the pixels of the first and the last column.  The first to
  // mark a root lists it, and for rho gives it its border pixel as value.
  {
    auto claim = [&](int run, int r, int x) {
      const int R = root_of(s, run);
      const uint32_t bit = 2u << (8 * (R & 3));
      const uint32_t was = atomicOr(reinterpret_cast<uint32_t*>(s.flag) + (R >> 2), bit);
      if (was & bit) return;
      s.pend[atomicAdd(&s.nlist, 1)] = (uint32_t)R;
      if (phi1 != nullptr) s.parent[R] = -((g.r0 + r) * g.W + 32 * g.w0 + x + 2);
    };
    const int rows = g.th > 1 ? 2 : 1;
    for (int i = tid; i < rows * g.tww + 2 * ns; i += blockDim.x) {
      if (i < rows * g.tww) {
        const int r = i < g.tww ? 0 : g.th - 1, w = i < g.tww ? i : i - g.tww, k = r >> 1;
        const uint32_t m = s.m[r][w];
        uint32_t rs = m & ~((m << 1) | (w > 0 ? (s.m[r][w - 1] >> 31) : 0u));
        const uint32_t st = s.st[k][w];
        const int id = s.base[k] + s.pre[k][w] - 1;
        while (rs) {
          const int p = __ffs(rs) - 1;
          rs &= rs - 1;
          claim(id + __popc(st & le_mask(p)), r, 32 * w + p);
        }
      } else {
        const int j = i - rows * g.tww, k = j >> 1;
        const int w = j & 1 ? g.tww - 1 : 0, p = j & 1 ? 31 : 0;
        for (int r = 2 * k; r <= 2 * k + 1; ++r)
          if ((s.m[r][w] >> p) & 1u)
            claim(s.base[k] + s.pre[k][w] + __popc(s.st[k][w] & le_mask(p)) - 1, r, 32 * w + p);
      }
    }
  }
  // 7. minimum pixel of each component (for canonical labels): only strip
  // runs in the component's first strip can hold it
  if (phi1 == nullptr) {
    for (int k = warp; k < ns; k += nw) {
      if (lane >= g.tww) continue;
      uint32_t sc = s.st[k][lane];
      while (sc) {
        const int p = __ffs(sc) - 1;
        sc &= sc - 1;
        const int x = 32 * lane + p;
        const int S = sid(s, k, x);
        const int R = root_of(s, S);
        if (R < s.base[k]) continue;
        // first pixel of the top row inside this strip run, else its start
        int best = -1;
        for (int ww = lane, pp = p; ww < g.tww; ++ww, pp = 0) {
          const uint32_t from = ~(le_mask(pp) >> 1);  // bits >= pp
          const uint32_t u = s.u[k][ww];
          // the run ends at the first zero of u or the next run start
          uint32_t stop = (~u | (s.st[k][ww] & ~(ww == lane ? le_mask(p) : 0u))) & from;
          if (ww == lane) stop &= ~(1u << p);
          const uint32_t ext = stop ? (from & ((stop & (0u - stop)) - 1u)) : from;
          const uint32_t hit = s.m[2 * k][ww] & ext;
          if (hit) { best = 32 * ww + __ffs(hit) - 1; break; }
          if (stop) break;
        }
        const int row = best >= 0 ? 2 * k : 2 * k + 1;
        const int col = best >= 0 ? best : x;
        atomicMax(&s.parent[R], -((g.r0 + row) * g.W + 32 * g.w0 + col + 2));
      }
    }
  }
  __syncthreads();
  return nruns;
}

// Keys of the component select.  A tile-local component is keyed by a border
// pixel v when it holds a seed pixel, and by v + npx when it does not; G then
// has 2 * npx entries.  The global merge links the larger root under the
// smaller, so a merged component's root is a seeded key (< npx) exactly when
// one of its parts was seeded: the seed flag travels with the union itself
// and no separate pass has to gather it.  (Components that do not reach the
// tile border need no key.)
VL_DEV int rz_key(int v, bool seeded, int npx) { return seeded ? v : v + npx; }

// The value of root R as G holds it: its key (rho) or its minimum pixel.
VL_DEV int root_key(const CclSmem& s, int R, bool rho, int npx) {
  const int v = -s.parent[R] - 2;
  return rho ? rz_key(v, s.flag[R] & 1, npx) : v;
}

// Publishes the tile's border in G: every border pixel points at its
// component's value, and so does the value itself.  The list of border roots
// goes to `list`: their number and that of strip runs, then value and run of
// each.
VL_DEV void ccl_publish(CclSmem& s, int nruns, const CclGeom& g, int32_t* G, bool rho, int npx,
                        int32_t* list) {
  const int nl = s.nlist;
  for (int i = threadIdx.x; i < nl; i += blockDim.x) {
    const int R = (int)s.pend[i], v = root_key(s, R, rho, npx);
    G[v] = v;
    list[2 + 2 * i] = v;
    list[3 + 2 * i] = R;
  }
  if (threadIdx.x == 0) {
    list[0] = nl;
    list[1] = nruns;
  }
  const int width = 32 * g.tww;
  const int n = 2 * width + 2 * g.th;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    int r, x;
    if (i < width) { r = 0; x = i; }
    else if (i < 2 * width) { r = g.th - 1; x = i - width; }
    else if (i < 2 * width + g.th) { r = i - 2 * width; x = 0; }
    else { r = i - 2 * width - g.th; x = width - 1; }
    const uint32_t m = s.m[r][x >> 5];
    if ((m >> (x & 31)) & 1u) {
      const int v = root_key(s, root_of(s, sid(s, r >> 1, x)), rho, npx);
      const int gid = (g.r0 + r) * g.W + 32 * g.w0 + x;
      if (gid != v) G[gid] = v;  // (the value's own entry is written above)
    }
  }
}

// Per-tile storage between the local and the final pass, in a tile's share of
// the scratch (ccl_tile_cap entries, an int32 and a byte each).
// Labels: s.parent of every strip run, then the list of border roots in the
// bytes.  Rho: a 16-bit code per strip run (RzSmem) in the first half of the
// words, the list in the second.  The final pass rebuilds the strips from
// the mask and reloads this instead of labelling the tile again.
VL_DEV int ccl_tile_cap(int Wp, int cth = CCL_TH) { return (cth / 2) * min(CCL_TWW, Wp) * 32; }

VL_DEV void ccl_tile_save(const CclSmem& s, int nruns, int32_t* tpar) {
  for (int i = threadIdx.x; i < nruns; i += blockDim.x) tpar[i] = s.parent[i];
}
VL_DEV void rz_tile_save(const CclSmem& s, int nruns, int32_t* tpar) {
  auto code = [&](int i) -> uint32_t {
    const int p = s.parent[i];
    return p >= 0 ? (uint32_t)p : RZ_ROOT | ((s.flag[i] & 1) ? RZ_SEED : 0u);
  };
  for (int i = 2 * threadIdx.x; i < nruns; i += 2 * blockDim.x)
    reinterpret_cast<uint32_t*>(tpar)[i >> 1] = code(i) | (i + 1 < nruns ? code(i + 1) : 0u) << 16;
}

// The final pass of labels up to the point where every root of s.parent holds
// its component's label: the walks in G of the border roots start first, and
// their latency passes beside the strips'.  Returns the number of strip runs
// or -1; a block barrier at the end.
VL_DEV int ccl_tile_load(CclSmem& s, const uint32_t* mask, const CclGeom& g, int conn,
                         const int32_t* tpar, const int32_t* list, int cap, int32_t* G, int npx,
                         int32_t* status) {
  const StripRows rows = ccl_load_rows(mask, g);
  const int2 head = __ldcg(reinterpret_cast<const int2*>(list));  // border roots, strip runs
  const int nl = min(head.x, min(CCL_MAXBORDER, cap / 8 - 1));
  for (int i = threadIdx.x; i < nl; i += blockDim.x) {
    const int2 e = __ldcg(reinterpret_cast<const int2*>(list) + 1 + i);
    s.pend[2 * i] = (uint32_t)e.y;
    s.pend[2 * i + 1] = (uint32_t)g_find(G, e.x, npx, status);
  }
  const int n = __shfl_sync(FULL, ccl_tile_strips(s, rows, nullptr, g, conn), 31);
  if (n > CCL_MAXRUNS) {
    set_status(status, ST_INTERNAL | RS_TRUNS);
    return -1;
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    int v = ldcg(tpar + i);
    if (v >= n) {  // never written by a successful local pass: keep indexes in range
      set_status(status, ST_INTERNAL | RS_TLOAD);
      v = -2;
    }
    s.parent[i] = v;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nl; i += blockDim.x) {
    const uint32_t R = s.pend[2 * i];
    if (R < (uint32_t)n) s.parent[R] = -((int)s.pend[2 * i + 1] + 2);
    else set_status(status, ST_INTERNAL | RS_TLOAD);
  }
  __syncthreads();
  return n;
}

// The final pass of rho: Z = the selected components of the tile.  A border
// component is selected when its root in G is a seeded key, any other when
// it holds a seed pixel.  cap: the tile's capacity (ccl_tile_cap).  The loads
// of rows, codes and list are in flight together, and the walks in G start
// before the strips are worked out.
VL_DEV void rz_tile_select(RzSmem& s, const uint32_t* mask, const CclGeom& g, int conn,
                           const int32_t* tpar, int cap, int32_t* G, int npx, uint32_t* Z,
                           int32_t* status) {
  const int tid = threadIdx.x, lane = tid & 31, k = tid >> 5;
  const int ns = (g.th + 1) >> 1;
  const StripRows rows = ccl_load_rows(mask, g);
  const int32_t* list = tpar + cap / 2;
  const int2 head = __ldcg(reinterpret_cast<const int2*>(list));  // border roots, strip runs
  const int nl = min(head.x, min(CCL_MAXBORDER, cap / 4 - 1));
  const int saved = min(head.y, min(CCL_MAXRUNS, cap));
  const uint32_t* codes = reinterpret_cast<const uint32_t*>(tpar);
  uint32_t* sc = reinterpret_cast<uint32_t*>(s.code);
  for (int i = tid; 2 * i < saved; i += blockDim.x) cp_async4(sc + i, codes + i);
  cp_async_commit();
  for (int i = tid; i < nl; i += blockDim.x) {
    const int2 e = __ldcg(reinterpret_cast<const int2*>(list) + 1 + i);
    const bool sel = g_find(G, e.x, 2 * npx, status) < npx;
    s.list[i] = (uint32_t)e.y | (sel ? RZ_SEL << 16 : 0u);
  }
  const int n = __shfl_sync(FULL, ccl_tile_strips(s, rows, nullptr, g, conn), 31);
  cp_async_wait<0>();
  if (n > CCL_MAXRUNS || n != saved) {  // (uniform) not the tile that was saved
    set_status(status, ST_INTERNAL | RS_TLOAD);
    return;
  }
  __syncthreads();
  for (int i = tid; i < nl; i += blockDim.x) {
    const uint32_t e = s.list[i], R = e & 0xFFFFu;
    if (R >= (uint32_t)n) set_status(status, ST_INTERNAL | RS_TLOAD);
    else if (e >> 16) s.code[R] |= RZ_SEL;
  }
  __syncthreads();
  auto selected = [&](int run) {
    uint32_t c = s.code[run];
    if (!(c & RZ_ROOT)) c = s.code[c & (CCL_MAXRUNS - 1)];
    return (c & (RZ_SEED | RZ_SEL)) != 0;
  };
  if (k < ns && lane < g.tww) {
    const uint32_t u = s.u[k][lane], st = s.st[k][lane];
    const int id = s.base[k] + s.pre[k][lane];
    uint32_t f = 0, runs = st;
    for (int j = 0; runs; ++j) {
      const uint32_t bit = runs & (0u - runs);
      runs ^= bit;
      if (selected(id + j)) f |= bit;
    }
    // a run entering from the left word continues through bit 0
    const uint32_t e = u & ~st;
    const uint32_t inj = (f << 1) | ((e & 1u) && selected(id - 1) ? 1u : 0u);
    // carry through the continuation bits of each selected run
    const uint32_t sel = f | (((e + inj) ^ e) & e);
    for (int r = 2 * k; r <= 2 * k + 1 && r < g.th; ++r)
      Z[(size_t)(g.r0 + r) * g.Wp + g.w0 + lane] = s.m[r][lane] & sel;
  }
}

// Write labels of the tile (after ccl_tile_load).  First every strip run takes
// its root's encoded value (after the flatten non-roots point at roots, and
// roots are not written, so the pass needs no ordering).  Then, where rows
// start on 16-byte boundaries, each lane writes 4 consecutive pixels per step,
// a warp 128 pixels of a row; elsewhere a lane writes one pixel of a word, so
// that a store of the warp still covers 128 bytes, for four words at a time.
// (Four stores a lane, 16 bytes apart from its neighbours', took 25 us for the
// whole pass at 3001 x 2777; so it takes 18.)
VL_DEV void ccl_write_labels(CclSmem& s, int nruns, const CclGeom& g, int32_t* labels) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;
  for (int i = threadIdx.x; i < nruns; i += blockDim.x) {
    const int p = s.parent[i];
    if (p >= 0) s.parent[i] = s.parent[p];
  }
  __syncthreads();
  const int x_end = min(32 * g.tww, g.W - 32 * g.w0);
  const bool vec = (g.W & 3) == 0;
  for (int r = warp; r < g.th; r += nw) {
    int32_t* row = labels + (size_t)(g.r0 + r) * g.W + 32 * g.w0;
    const int k = r >> 1;
    if (vec) {
      for (int x0 = 4 * lane; x0 < x_end; x0 += 128) {
        const int w = x0 >> 5, b = x0 & 31;
        const uint32_t bits = s.m[r][w] >> b;
        const uint32_t st = s.st[k][w];
        const int base = s.base[k] + s.pre[k][w] - 1;
        int v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          v[q] = ((bits >> q) & 1u) ? -s.parent[base + __popc(st & le_mask(b + q))] - 2 : -1;
        *reinterpret_cast<int4*>(row + x0) = make_int4(v[0], v[1], v[2], v[3]);
      }
    } else {
      const uint32_t le = le_mask(lane);
      for (int w = 0; 32 * w < x_end; w += 4) {  // (tiles have whole vectors of words)
        int v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int base = s.base[k] + s.pre[k][w + q] - 1;
          v[q] = (s.m[r][w + q] >> lane) & 1u ? -s.parent[base + __popc(s.st[k][w + q] & le)] - 2 : -1;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (32 * (w + q) + lane < x_end) row[32 * (w + q) + lane] = v[q];
      }
    }
  }
}

// --------------------------------------------------------- border merge --
// The borders between labelling tiles are merged by a pass of their own
// after the labelling launch, in merge units: one per word of each
// horizontal tile border (its 32 columns) and one per 32 rows of each
// vertical tile border.  A warp takes a unit, one lane per column (or row),
// so the unions of a unit run side by side.  (A merge inside the labelling
// launch, by whichever tile beside a border finished last, measured slower:
// its latency-bound walks then hold a labelling CTA instead of running at
// full occupancy.)

// Which of columns x-1, x, x+1 (8-adjacency) or x (4-adjacency) of a row is
// set, leftmost first, as an offset -1/0/1 (2: none).  The row is given by
// the words left of, at, and right of x's word (0 outside the image), and
// b = x mod 32.
VL_DEV int window_hit(uint32_t l, uint32_t c, uint32_t r, int b, int conn) {
  if (conn == 8) {
    const uint32_t left = b > 0 ? (c >> (b - 1)) & 1u : (l >> 31);
    if (left) return -1;
    if ((c >> b) & 1u) return 0;
    const uint32_t right = b < 31 ? (c >> (b + 1)) & 1u : (r & 1u);
    return right ? 1 : 2;
  }
  return ((c >> b) & 1u) ? 0 : 2;
}

// Every lane offers at most one pixel pair (a, b) across a tile border.  The
// pairs become pairs of component keys (border pixels hold their component's
// representative in G, so a plain read gives a key without a find); equal
// key pairs in the warp are united once, by the lowest lane holding them.
// Must be called by the whole warp.
VL_DEV void warp_unite(int32_t* G, bool valid, int a, int b, int glen, int32_t* status) {
  int ka = 0, kb = 0;
  if (valid) {
    ka = ldcg(&G[a]);
    kb = ldcg(&G[b]);
    valid = ka != kb;
  }
  const unsigned long long key =
      valid ? (((unsigned long long)(unsigned)max(ka, kb) << 32) | (unsigned)min(ka, kb)) : ~0ull;
  const unsigned peers = __match_any_sync(FULL, key);
  if (valid && (threadIdx.x & 31) == __ffs(peers) - 1) g_union(G, ka, kb, glen, status);
}

// Two pairs per lane, (a1, b1) and (a2, b2).  When the warp holds at most 32
// valid pairs they are dealt out one per lane, so the unions run side by
// side in one round instead of two.  Must be called by the whole warp.
VL_DEV void warp_unite2(int32_t* G, bool v1, int a1, int b1, bool v2, int a2, int b2, int glen,
                        int32_t* status) {
  const int lane = threadIdx.x & 31;
  const unsigned m1 = __ballot_sync(FULL, v1), m2 = __ballot_sync(FULL, v2);
  const int n1 = __popc(m1), n = n1 + __popc(m2);
  if (n > 32) {
    warp_unite(G, v1, a1, b1, glen, status);
    warp_unite(G, v2, a2, b2, glen, status);
    return;
  }
  // lane L takes the L-th valid pair: the first kind's in lane order, then
  // the second's
  int src = lane;
  if (lane < n1) src = __fns(m1, 0, lane + 1);
  else if (lane < n) src = __fns(m2, 0, lane - n1 + 1);
  const int xa1 = __shfl_sync(FULL, a1, src), xb1 = __shfl_sync(FULL, b1, src);
  const int xa2 = __shfl_sync(FULL, a2, src), xb2 = __shfl_sync(FULL, b2, src);
  const bool first = lane < n1;
  warp_unite(G, lane < n, first ? xa1 : xa2, first ? xb1 : xb2, glen, status);
}

// Unite the components of row yu and row yd (rows of the stored image) that
// touch in word w: with conn 8 a pixel meets the three pixels at x - 1, x,
// x + 1 of the other row, with conn 4 only the one at x.  Every row-run
// start of either row is checked against that window of the other row: two
// runs that touch always have a start of one run inside the other's window.
// Padding bits are cleared.  Must be called by the whole warp.
VL_DEV void ccl_merge_rows(const uint32_t* m, int W, int Wp, int yu, int yd, int w, int conn,
                           int32_t* G, int glen, int32_t* status) {
  const int lane = threadIdx.x & 31;
  uint32_t v = 0;
  if (lane < 6) {
    const int ww = w - 1 + lane % 3;
    if (ww >= 0 && ww < Wp) v = ldcg(&m[(size_t)(lane < 3 ? yu : yd) * Wp + ww]) & vmask(ww, W);
  }
  const uint32_t mul = __shfl_sync(FULL, v, 0), mu = __shfl_sync(FULL, v, 1),
                 mur = __shfl_sync(FULL, v, 2), mdl = __shfl_sync(FULL, v, 3),
                 md = __shfl_sync(FULL, v, 4), mdr = __shfl_sync(FULL, v, 5);
  const uint32_t sd = md & ~((md << 1) | (mdl >> 31));
  const uint32_t su = mu & ~((mu << 1) | (mul >> 31));
  const int x = 32 * w + lane;
  const int dd = (sd >> lane) & 1u ? window_hit(mul, mu, mur, lane, conn) : 2;
  const int du = (su >> lane) & 1u ? window_hit(mdl, md, mdr, lane, conn) : 2;
  warp_unite2(G, dd != 2, yd * W + x, yu * W + x + dd, du != 2, yu * W + x, yd * W + x + du,
              glen, status);
}

// (Hs: slice rows of a volume, H for an image; horizontal borders are those
// between the tile rows of one slice.)
VL_DEV int merge_units(int H, int Wp, int tiles_x, int Hs, int cth = CCL_TH) {
  const int tys = (Hs + cth - 1) / cth;
  return (H / Hs) * (tys - 1) * Wp + (tiles_x - 1) * ((H + 31) >> 5);
}

// Unite the components that touch across the tile border of merge unit
// `unit`.  A horizontal border is ccl_merge_rows over the whole row.  A
// vertical border pairs each set pixel left of it with the pixel right of it,
// or, for 8-adjacency when that one is clear, with its diagonal neighbours
// (both border columns lie inside the image: a tile border is a multiple of
// 1024 columns, below W).  Must be called by the whole warp.
VL_DEV void ccl_merge_unit(const uint32_t* m, int H, int W, int Wp, int unit, int conn,
                           int32_t* G, int glen, int32_t* status, int Hs, int cth = CCL_TH) {
  const int lane = threadIdx.x & 31;
  const int tys = (Hs + cth - 1) / cth;
  const int nh = (H / Hs) * (tys - 1) * Wp;
  if (unit < nh) {
    const int border = unit / Wp, w = unit - border * Wp;  // border: over all slices
    const int z = border / (tys - 1), k = border - z * (tys - 1) + 1;
    const int yd = z * Hs + k * cth, yu = yd - 1;
    ccl_merge_rows(m, W, Wp, yu, yd, w, conn, G, glen, status);
  } else {
    const int nv = (H + 31) >> 5;
    const int j = unit - nh;
    const int kk = j / nv + 1;
    const int y = (j - (kk - 1) * nv) * 32 + lane;
    const int x0 = kk * CCL_TWW * 32;  // first column right of the border (< W)
    const int wl = (x0 - 1) >> 5, wr = x0 >> 5;
    uint32_t L = 0, R = 0, Ru = 0, Rd = 0;
    if (y < H) {
      L = ldcg(&m[(size_t)y * Wp + wl]) >> 31;
      R = ldcg(&m[(size_t)y * Wp + wr]) & 1u;
    }
    if (conn == 8) {
      Ru = __shfl_up_sync(FULL, R, 1);
      Rd = __shfl_down_sync(FULL, R, 1);
      if (lane == 0) Ru = (y > 0 && y - 1 < H) ? ldcg(&m[(size_t)(y - 1) * Wp + wr]) & 1u : 0u;
      if (lane == 31) Rd = (y + 1 < H) ? ldcg(&m[(size_t)(y + 1) * Wp + wr]) & 1u : 0u;
      // diagonals stay inside one slice of a volume
      if (y % Hs == 0) Ru = 0;
      if ((y + 1) % Hs == 0) Rd = 0;
    }
    // (lane-dependent choices go into the arguments: every lane calls)
    const int a = y * W + x0 - 1;
    const bool straight = R || conn == 4;
    warp_unite2(G, L && (straight ? R : Ru), a, (straight ? y : y - 1) * W + x0,
                L && !straight && Rd, a, (y + 1) * W + x0, glen, status);
  }
}

}  // namespace vl
