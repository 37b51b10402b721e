// Volumes: the logic of Sec. 2 on D x H x W voxel grids, the paper's outlook
// beyond 2D slices (Sec. 1 and Sec. 5).  A volume is stored as its D slices
// stacked into one image of D * H rows (slice z is rows [z * H, (z + 1) * H)),
// bit-packed like any mask, so thresholds, not/and and percentiles run the
// 2D kernels unchanged.  Only the operators that look at neighbours differ:
//   N   -- 26-adjacency: the 3 x 3 x 3 cube, i.e. the 2D 3 x 3 dilation of the
//          OR of the rows y-1..y+1 of slices z-1..z+1; 6-adjacency: the faces,
//          i.e. the 2D cross of slice z OR the same word of slices z-1, z+1.
//          Both clip at the volume's border (no voxels outside it).
//   CCL -- 2D labelling of every slice (tiles never straddle slices; the
//          in-slice adjacency is 8 for 26 and 4 for 6), then a merge between
//          neighbouring slices: the rows (z, y) and (z + 1, y + dy) with
//          dy in {-1, 0, 1} under a 3-voxel window (26), or (z, y) and
//          (z + 1, y) voxel on voxel (6); then every voxel takes its root.
//          Labels are canonical: the minimum linear index z*H*W + y*W + x.
//   rho -- as for images (Sec. 3.2): rho phi1[phi2] = N(phi1 or Z), Z the
//          phi2-components that meet N phi1; Z from the phi2-components' union-find,
//          a flag per root set from the seed voxels.
#include "dev_ccl.cuh"
#include "dev_common.cuh"
#include "kernels.h"
#include "launch.cuh"

namespace vl {

namespace {

constexpr int kThreads = 256;

int grid_for(long long items, int per_block, int cap = 152 * 32) {
  long long b = (items + per_block - 1) / per_block;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (int)b;
}

// Word w of row `row` of the stored image, 0 outside [0, Wp).
VL_DEV uint32_t word_at(const uint32_t* a, int Wp, int row, int w) {
  return (w >= 0 && w < Wp) ? __ldg(a + (size_t)row * Wp + w) : 0u;
}

// N a on word w of row y of the stored image.
VL_DEV uint32_t near3_word(const uint32_t* a, const MaskGeom& g, int conn, int y, int w) {
  const int Hs = slice_rows(g), D = g.H / Hs;
  const int z = y / Hs, yz = y - z * Hs;
  uint32_t res;
  if (conn == 26) {
    uint32_t l = 0, c = 0, r = 0;  // OR of the 9 rows around, per column word
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy) {
        if (z + dz < 0 || z + dz >= D || yz + dy < 0 || yz + dy >= Hs) continue;
        const int row = y + dz * Hs + dy;
        l |= word_at(a, g.Wp, row, w - 1);
        c |= word_at(a, g.Wp, row, w);
        r |= word_at(a, g.Wp, row, w + 1);
      }
    res = hdil(l, c, r);
  } else {
    res = hdil(word_at(a, g.Wp, y, w - 1), word_at(a, g.Wp, y, w), word_at(a, g.Wp, y, w + 1));
    if (yz > 0) res |= word_at(a, g.Wp, y - 1, w);
    if (yz + 1 < Hs) res |= word_at(a, g.Wp, y + 1, w);
    if (z > 0) res |= word_at(a, g.Wp, y - Hs, w);
    if (z + 1 < D) res |= word_at(a, g.Wp, y + Hs, w);
  }
  return res & vmask(w, g.W);
}

// N a on whole vectors of four words, one a thread: nine vector loads and the
// words beside them instead of 27 loads a word.
__global__ void __launch_bounds__(kThreads) k_near3(const uint32_t* a, MaskGeom g, int conn, uint4* out) {
  grid_wait(a);
  const int nv = g.Wp >> 2, Hs = slice_rows(g), D = g.H / Hs;
  const long long n = (long long)g.H * nv;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    int y, jv, z, yz;
    split_index(i, nv, y, jv);
    split_index(y, Hs, z, yz);
    const bool left = jv > 0, right = jv + 1 < nv;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    // row (dy, dz) away, and the words beside its vector
    auto inside = [&](int dy, int dz) {
      return z + dz >= 0 && z + dz < D && yz + dy >= 0 && yz + dy < Hs;
    };
    auto at = [&](int dy, int dz) { return a + 4 * i + (long long)(dz * Hs + dy) * g.Wp; };
    uint4 x = zero, o = zero;
    uint32_t l = 0, e = 0;
    if (conn == 26) {
#pragma unroll
      for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
          if (inside(dy, dz)) {
            const uint32_t* p = at(dy, dz);
            x = or4(x, __ldg(reinterpret_cast<const uint4*>(p)));
            if (left) l |= __ldg(p - 1);
            if (right) e |= __ldg(p + 4);
          }
    } else {
      const uint32_t* p = at(0, 0);
      x = __ldg(reinterpret_cast<const uint4*>(p));
      if (left) l = __ldg(p - 1);
      if (right) e = __ldg(p + 4);
      if (inside(-1, 0)) o = or4(o, __ldg(reinterpret_cast<const uint4*>(at(-1, 0))));
      if (inside(1, 0)) o = or4(o, __ldg(reinterpret_cast<const uint4*>(at(1, 0))));
      if (inside(0, -1)) o = or4(o, __ldg(reinterpret_cast<const uint4*>(at(0, -1))));
      if (inside(0, 1)) o = or4(o, __ldg(reinterpret_cast<const uint4*>(at(0, 1))));
    }
    out[i] = clip_vec(near_vec(x, o, l, e), jv, g.W);
  }
}

// Word w of row yz of slice z, without padding; 0 outside the volume.
struct SliceRows {
  const uint32_t* m;
  int W, Wp, Hs, w;
  uint32_t edge[3];  // pixels of words w - 1, w, w + 1 inside the image
  VL_DEV SliceRows(const uint32_t* m_, const MaskGeom& g, int w_)
      : m(m_), W(g.W), Wp(g.Wp), Hs(slice_rows(g)), w(w_) {
    edge[0] = w > 0 ? FULL : 0u;
    edge[1] = vmask(w, W);
    edge[2] = w + 1 < Wp ? vmask(w + 1, W) : 0u;
  }
  VL_DEV uint32_t at(int z, int yz, int d) const {
    return yz >= 0 && yz < Hs && edge[d + 1]
               ? __ldg(m + (size_t)(z * Hs + yz) * Wp + w + d) & edge[d + 1] : 0u;
  }
};

// Bits of `hit` spread down through the runs of c they lie in.
VL_DEV uint32_t fill_down(uint32_t hit, uint32_t c) {
  uint32_t t = hit & c, p = c;
#pragma unroll
  for (int o = 1; o < 32; o *= 2) {
    t |= p & (t >> o);
    p &= p >> o;
  }
  return t;
}

// The pairs of voxels (p, q) of word i of a slice and of the slice behind it
// that have to be united, handed to f.
template <class F>
VL_DEV void zmerge_word(const uint32_t* m, const MaskGeom& g, int conn, long long i, F f) {
  const int Hs = slice_rows(g);
  int row, w, z, yz;
  split_index(i, g.Wp, row, w);
  split_index(row, Hs, z, yz);
  const SliceRows R(m, g, w);
  const uint32_t a = R.at(z, yz, 0);
  if (!a) return;
  const int p0 = row * g.W + 32 * w, q0 = p0 + Hs * g.W;  // first voxels of the words
  auto unite = [&](uint32_t set, int dq) {
    while (set) {
      const int b = __ffs(set) - 1;
      set &= set - 1;
      f(p0 + b, q0 + b + dq);
    }
  };
  const uint32_t b0 = R.at(z + 1, yz, 0), c = a & b0;
  const uint32_t al = R.at(z, yz, -1), bl = R.at(z + 1, yz, -1);
  const uint32_t au = R.at(z, yz - 1, 0), bu = R.at(z + 1, yz - 1, 0);
  uint32_t cu = au & bu;  // contacts of the row above
  if (conn == 26) cu |= (cu << 1) | (cu >> 1);
  const uint32_t starts = c & ~((c << 1) | ((al & bl) >> 31));
  unite(starts & ~fill_down(cu, c), 0);
  if (conn != 26) return;
  const uint32_t p = a & ~b0;
  if (!p) return;
  const uint32_t ar = R.at(z, yz, 1), br = R.at(z + 1, yz, 1);
  // same row, one column apart
  const uint32_t q = b0 & ~a;
  unite(p & ((q << 1) | ((bl & ~al) >> 31)), -1);
  unite(p & ((q >> 1) | ((br & ~ar) << 31)), 1);
  const uint32_t a_left = (a << 1) | (al >> 31), a_right = (a >> 1) | (ar << 31);
#pragma unroll
  for (int dy = -1; dy <= 1; dy += 2) {
    const uint32_t ay = dy < 0 ? au : R.at(z, yz + 1, 0), by = dy < 0 ? bu : R.at(z + 1, yz + 1, 0);
    const uint32_t qy = by & ~ay;
    const uint32_t over = p & qy;
    unite(over & ~(over << 1), dy * g.W);
    const uint32_t free = p & ~by;
    if (!free) continue;
    const uint32_t qyl = R.at(z + 1, yz + dy, -1) & ~R.at(z, yz + dy, -1);
    const uint32_t qyr = R.at(z + 1, yz + dy, 1) & ~R.at(z, yz + dy, 1);
    unite(free & ~a_left & ((qy << 1) | (qyl >> 31)), dy * g.W - 1);
    unite(free & ~a_right & ((qy >> 1) | (qyr << 31)), dy * g.W + 1);
  }
}

// Unite the components of slices z and z + 1; one thread per word of slice z.
// L holds, for every voxel of the mask, its slice component's key (after the
// 2D pass: the component's minimum index, which is a root).
//
// What costs is the unions, each a chain of dependent loads, so the voxel
// pairs (p, q) across the slices are thinned out with bit operations until
// one or two per contact remain.  Straight pairs (p over q): of every run of
// contacts in a row one is taken, and none when the run touches a contact of
// the row above (p and q are then connected inside their slices to a pair
// taken there).  Pairs of neighbours that are not straight (26-adjacency)
// count only where neither voxel has a straight contact (else q, or p, is a
// slice neighbour of that contact); one row apart, diagonal ones only where
// the voxel beside p in its row and the one beside q in its own are clear
// (else that one makes a pair one column closer), and of neighbouring pairs
// in the same direction the first.  (A warp per row that offered every run
// start of either row took 147 to 284 us on a 155 x 240 x 240 scan; this
// takes 16 to 51.)
//
// Pairs go to a list of the block's and are dealt out to its threads from
// there: a thread that united those of its own word kept the others waiting
// where the mask is dense (48 to 116 us).
constexpr int ZMERGE_LIST = 3072;
__global__ void __launch_bounds__(kThreads) k_zmerge(const uint32_t* m, MaskGeom g, int conn, int32_t* L,
                                                     int32_t* status) {
  __shared__ int2 list[ZMERGE_LIST];
  __shared__ int listed;
  grid_wait(m);
  const int Hs = slice_rows(g), D = g.H / Hs;
  const int npx = g.H * g.W;
  const long long n = (long long)(D - 1) * Hs * g.Wp;
  auto pair = [&](int p, int q) {
    const int ka = ldcg(&L[p]), kb = ldcg(&L[q]);
    if (ka != kb) g_union(L, ka, kb, npx, status);
  };
  for (long long base = (long long)blockIdx.x * blockDim.x; base < n;
       base += (long long)gridDim.x * blockDim.x) {
    if (threadIdx.x == 0) listed = 0;
    __syncthreads();
    const long long i = base + threadIdx.x;
    if (i < n)
      zmerge_word(m, g, conn, i, [&](int p, int q) {
        const int at = atomicAdd(&listed, 1);
        if (at < ZMERGE_LIST) list[at] = make_int2(p, q);
        else pair(p, q);
      });
    __syncthreads();
    const int k = min(listed, ZMERGE_LIST);
    for (int j = threadIdx.x; j < k; j += blockDim.x) pair(list[j].x, list[j].y);
    __syncthreads();
  }
}

// Every voxel of the mask takes the root of its key (finds compress: a
// node only moves to an ancestor, and the root is the label of every node
// on the way).
__global__ void k_relabel(const uint32_t* m, MaskGeom g, int32_t* L, int32_t* status) {
  grid_wait(m);
  const int npx = g.H * g.W;
  // grid-stride over the voxels, row and column stepped instead of divided
  const int stride = gridDim.x * blockDim.x;
  const int sy = stride / g.W, sx = stride - sy * g.W;
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int y, x;
  split_index(i, g.W, y, x);
  for (; i < npx; i += stride) {
    if ((__ldg(m + (size_t)y * g.Wp + (x >> 5)) >> (x & 31)) & 1u)
      L[i] = g_find(L, ldcg(&L[i]), npx, status);
    y += sy;
    x += sx;
    if (x >= g.W) { x -= g.W; ++y; }
  }
}

// Runs of the words of a block (at most 16 a word), dealt out to its threads:
// each run is a walk through the union-find, and one word may hold many.  (With
// each thread walking its own word's runs, the seeds of a 155 x 240 x 240 scan
// took 25 us and the selection 19; so they take 18 and 13.)
struct BlockRuns {
  int first[kThreads];        // first voxel of each thread's word
  uint16_t run[16 * kThreads];  // thread << 5 | bit
  int n;
};
// Lists the bits of `starts` of this thread's word; block barriers around.
VL_DEV int list_runs(BlockRuns& s, int first, uint32_t starts) {
  const int t = threadIdx.x;
  if (t == 0) s.n = 0;
  s.first[t] = first;
  __syncthreads();
  if (starts) {
    int at = atomicAdd(&s.n, __popc(starts));
    while (starts) {
      s.run[at++] = (uint16_t)(t << 5 | (__ffs(starts) - 1));
      starts &= starts - 1;
    }
  }
  __syncthreads();
  return s.n;
}

// F[root] = 1 for the component of every seed, i.e. voxel of phi2 in N phi1
// (benign races: every writer writes 1).  Seeds lie in phi2, so the voxels of
// a run of seeds share one component: only the first voxel of every run is
// looked up.  The union-find is walked from the voxel's key: labels of all
// voxels would be a pass over the volume for these few.
__global__ void __launch_bounds__(kThreads) k_seed_flags(const uint32_t* phi1, const uint32_t* phi2,
                                                         MaskGeom g, int conn, int32_t* L, uint8_t* F,
                                                         int32_t* status) {
  __shared__ BlockRuns s;
  grid_wait(phi1, phi2);
  const long long nwords = (long long)g.H * g.Wp;
  const int npx = g.H * g.W;
  for (long long base = (long long)blockIdx.x * kThreads; base < nwords;
       base += (long long)gridDim.x * kThreads) {
    const long long i = base + threadIdx.x;
    int y = 0, w = 0;
    uint32_t starts = 0;
    if (i < nwords) {
      split_index(i, g.Wp, y, w);
      const uint32_t m = __ldg(phi2 + i) & vmask(w, g.W);
      if (m) {
        const uint32_t seeds = near3_word(phi1, g, conn, y, w) & m;
        starts = seeds & ~(seeds << 1);
      }
    }
    const int n = list_runs(s, y * g.W + 32 * w, starts);
    for (int j = threadIdx.x; j < n; j += kThreads) {
      const int v = s.first[s.run[j] >> 5] + (s.run[j] & 31);
      const int root = g_find(L, ldcg(&L[v]), npx, status);
      if (!__ldcg(F + root)) F[root] = 1;
    }
    __syncthreads();
  }
}

// Z = the voxels of phi2 whose component is flagged: one lookup per run of
// phi2 inside the word (a run is one component), the run's bits taken whole.
__global__ void __launch_bounds__(kThreads) k_select_flagged(const uint32_t* phi2, MaskGeom g, int32_t* L,
                                                             const uint8_t* F, uint32_t* Z,
                                                             int32_t* status) {
  __shared__ BlockRuns s;
  __shared__ uint32_t words[kThreads], sel[kThreads];
  grid_wait(phi2, F);
  const long long nwords = (long long)g.H * g.Wp;
  const int npx = g.H * g.W;
  for (long long base = (long long)blockIdx.x * kThreads; base < nwords;
       base += (long long)gridDim.x * kThreads) {
    const long long i = base + threadIdx.x;
    int y = 0, w = 0;
    uint32_t bits = 0;
    if (i < nwords) {
      split_index(i, g.Wp, y, w);
      bits = __ldg(phi2 + i) & vmask(w, g.W);
    }
    words[threadIdx.x] = bits;
    sel[threadIdx.x] = 0;
    const int n = list_runs(s, y * g.W + 32 * w, bits & ~(bits << 1));
    for (int j = threadIdx.x; j < n; j += kThreads) {
      const int t = s.run[j] >> 5, b = s.run[j] & 31;
      const int root = g_find(L, ldcg(&L[s.first[t] + b]), npx, status);
      if (!__ldg(F + root)) continue;
      // the run: bits b.. up to the first clear bit
      const uint32_t from = words[t] >> b;
      const uint32_t run = ~from ? ((~from & (0u - ~from)) - 1u) : 0xFFFFFFFFu;
      atomicOr(&sel[t], run << b);
    }
    __syncthreads();
    if (i < nwords) Z[i] = sel[threadIdx.x];
  }
}

}  // namespace

cudaError_t launch_near3(const uint32_t* a, MaskGeom g, int conn, uint32_t* out, cudaStream_t st) {
  return launch_early(k_near3, grid_for((long long)g.H * (g.Wp >> 2), kThreads), kThreads, 0, st, a, g,
                      conn, reinterpret_cast<uint4*>(out));
}

// The union-find of a volume's components: every voxel's key leads to its
// component's root, the minimum index of all its voxels.
static cudaError_t launch_components3(const uint32_t* mask, MaskGeom g, int conn, CclScratch sc,
                                      int32_t* status, cudaStream_t st) {
  cudaError_t e = launch_ccl_labels(mask, g, conn == 26 ? 8 : 4, sc, status, st);
  if (e) return e;
  const int Hs = slice_rows(g), D = g.H / Hs;
  if (D < 2) return cudaSuccess;
  const long long words = (long long)(D - 1) * Hs * g.Wp;
  return launch_early(k_zmerge, grid_for(words, kThreads), kThreads, 0, st, mask, g, conn, sc.G, status);
}

cudaError_t launch_labels3(const uint32_t* mask, MaskGeom g, int conn, CclScratch sc,
                           int32_t* status, cudaStream_t st) {
  cudaError_t e = launch_components3(mask, g, conn, sc, status, st);
  if (e || g.H == slice_rows(g)) return e;
  return launch_early(k_relabel, grid_for((long long)g.H * g.W, kThreads * 4), kThreads, 0, st, mask, g,
                      sc.G, status);
}

cudaError_t launch_rz3(const uint32_t* phi1, const uint32_t* phi2, MaskGeom g, int conn,
                       Rz3Scratch sc, uint32_t* Z, int32_t* status, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(sc.F, 0, (size_t)g.H * g.W, st);
  if (!e) e = launch_components3(phi2, g, conn, sc.ccl, status, st);
  if (e) return e;
  const long long nwords = (long long)g.H * g.Wp;
  e = launch_early(k_seed_flags, grid_for(nwords, kThreads), kThreads, 0, st, phi1, phi2, g, conn,
                   sc.ccl.G, sc.F, status);
  if (e) return e;
  return launch_early(k_select_flagged, grid_for(nwords, kThreads), kThreads, 0, st, phi2, g, sc.ccl.G,
                      sc.F, Z, status);
}

}  // namespace vl
