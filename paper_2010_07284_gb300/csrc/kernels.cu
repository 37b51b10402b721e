// Plain per-operator kernels: one launch per primitive over a whole image.
// They are the baseline execution form and the building blocks of vl_ccl.
#include <algorithm>
#include <mutex>

#include "dev_ccl.cuh"
#include "dev_common.cuh"
#include "dev_select.cuh"
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

// ------------------------------------------------------------ pointwise --

// N thresholds of one channel (rows of 32 * Wp elements) in one pass.  A lane
// loads 4 pixels (16 bytes, or 8 of uint16) four times, so that a warp covers
// 16 words and has four loads in flight a lane; three shuffles a threshold
// put them together.  Bound by memory: on the 36 MB of
// a 155 x 240 x 240 float channel 9.5 us for one threshold and 10.7 us for two
// (3.8 TB/s, launch included), where one pass each with two loads in flight
// and twelve shuffles took 15 us a threshold.
template <int N>
__global__ void __launch_bounds__(kThreads) k_thresholds(const void* plane, int format,
                                                         MaskGeom g, const __grid_constant__ ThrSet T) {
  grid_wait(plane);
  float t[N];
#pragma unroll
  for (int k = 0; k < N; ++k) t[k] = T.job[k].t_dev ? __ldcg(T.job[k].t_dev) : T.job[k].t;
  const int lane = threadIdx.x & 31, sub = lane & 7, group = lane >> 3;
  const long long nwords = (long long)g.H * g.Wp;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  for (long long base = wid * 16; base < nwords; base += nwarps * 16) {
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long long i = base + 4 * u + group;
      v[u] = i < nwords ? ld_px4(plane, format, true, (size_t)i * 32 + 4 * sub)
                        : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const long long i = base + 4 * (sub >> 1) + group;  // the word this lane ends up with
    int y, w;
    split_index(i, g.Wp, y, w);
    const uint32_t keep = vmask(w, g.W);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      uint32_t n[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        n[u] = T.job[k].lt ? (v[u].x < t[k]) | (v[u].y < t[k]) << 1 | (v[u].z < t[k]) << 2 | (v[u].w < t[k]) << 3
                           : (v[u].x > t[k]) | (v[u].y > t[k]) << 1 | (v[u].z > t[k]) << 2 | (v[u].w > t[k]) << 3;
      const uint32_t word = join_nibbles4(n, sub);
      if (!(sub & 1) && i < nwords) T.job[k].out[i] = word & keep;
    }
  }
}

// Masks are rows of Wp / 4 vectors of four words; a thread takes one at a time
// (a word at a time, NOT took 5.3 us on 155 x 240 x 240 and takes 3.4).
template <int OP>  // 0 not, 1 and, 2 or, 3 const false, 4 const true, 5 and-not
__global__ void k_pointwise(const uint4* a, const uint4* b, MaskGeom g,
                            uint4* out) {
  grid_wait(a, b);
  const int nv = g.Wp >> 2;
  const long long n = (long long)g.H * nv;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    uint4 v = make_uint4(0u, 0u, 0u, 0u), x = v;
    if (OP == 0 || OP == 1 || OP == 2 || OP == 5) v = __ldg(a + i);
    if (OP == 1 || OP == 2 || OP == 5) x = __ldg(b + i);
    if (OP == 0 || OP == 4) {
      int y, jv;
      split_index(i, nv, y, jv);
      v = clip_vec(make_uint4(~v.x, ~v.y, ~v.z, ~v.w), jv, g.W);
    } else if (OP == 1) {
      v = make_uint4(v.x & x.x, v.y & x.y, v.z & x.z, v.w & x.w);
    } else if (OP == 2) {
      v = or4(v, x);
    } else if (OP == 5) {
      v = make_uint4(v.x & ~x.x, v.y & ~x.y, v.z & ~x.z, v.w & ~x.w);
    }
    out[i] = v;
  }
}

__global__ void k_near(const uint32_t* a, MaskGeom g, int conn, uint4* out) {
  grid_wait(a);
  const int nv = g.Wp >> 2;
  const long long n = (long long)g.H * nv;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    int y, jv;
    split_index(i, nv, y, jv);
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    const uint32_t* p = a + 4 * i;
    const bool up = y > 0, down = y + 1 < g.H, left = jv > 0, right = jv + 1 < nv;
    const uint4* v = reinterpret_cast<const uint4*>(p);
    const uint4 m = __ldg(v), u = up ? __ldg(v - nv) : zero, d = down ? __ldg(v + nv) : zero;
    uint32_t l = left ? __ldg(p - 1) : 0u, e = right ? __ldg(p + 4) : 0u;
    if (conn == 8) {
      if (left && up) l |= __ldg(p - g.Wp - 1);
      if (left && down) l |= __ldg(p + g.Wp - 1);
      if (right && up) e |= __ldg(p - g.Wp + 4);
      if (right && down) e |= __ldg(p + g.Wp + 4);
    }
    const uint4 o = or4(u, d), x = conn == 8 ? or4(m, o) : m;
    out[i] = clip_vec(near_vec(x, o, l, e), jv, g.W);
  }
}

// --------------------------------------------------------------- select --

// Percentile selects, many blocks each: block (x, y) takes its share of pass
// `pass` of select y; then one block per select.
constexpr int SEL_BATCH = 24;
struct SelBatch {
  SelJob job[SEL_BATCH];
  uint32_t* state;
  int H, W, pitch;
};
__global__ void __launch_bounds__(EXEC_THREADS, 2)
k_sel_pass(const __grid_constant__ SelBatch B, int pass) {
  __shared__ __align__(16) SelectSmem s;
  SelJob j = B.job[blockIdx.y];
  grid_wait(j.plane);
  sel_pass(s, SelChan{j.plane, j.format, 1, B.H, B.W, B.pitch}, pass, blockIdx.x, gridDim.x, j.rank,
           B.state + (size_t)blockIdx.y * SEL_HIST);
}
__global__ void __launch_bounds__(EXEC_THREADS) k_sel_finish(const __grid_constant__ SelBatch B) {
  __shared__ __align__(16) SelectSmem s;
  SelJob j = B.job[blockIdx.x];
  grid_wait(j.plane);
  const float v = sel_finish(s, B.state + (size_t)blockIdx.x * SEL_HIST,
                             SelChan{j.plane, j.format, 1, B.H, B.W, B.pitch}, j.rank);
  if (threadIdx.x == 0) *j.out = v;
}

// ----------------------------------------------------------- arithmetic --

// out = a (op) b pixel by pixel over H x W (row pitch `pitch` elements); b
// is a plane or, when null, the constant c.  One IEEE rounding per pixel.
__global__ void k_arith(int op, const void* a, int a_format, const void* b,
                        int b_format, float c, float* out, int H, int W, int pitch) {
  grid_wait(a, b);
  const long long n = (long long)H * W;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    int y, x;
    split_index(i, W, y, x);
    const size_t off = (size_t)y * pitch + x;
    const float u = ld_px(a, a_format, false, off);
    const float w = b ? ld_px(b, b_format, false, off) : c;
    float z;
    switch (op) {
      case A_ADD: z = __fadd_rn(u, w); break;
      case A_SUB: z = __fsub_rn(u, w); break;
      case A_MUL: z = __fmul_rn(u, w); break;
      default: z = __fdiv_rn(u, w); break;
    }
    out[off] = z;
  }
}

// ------------------------------------------------------------------ ccl --

// phi1 null: full labelling (canonical minimum pixels), else the select of rho.
__global__ void __launch_bounds__(EXEC_THREADS, 2)
k_ccl_local(const uint32_t* mask, const uint32_t* phi1, MaskGeom g, int tiles_x, int conn,
            CclScratch sc, int32_t* status) {
  grid_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CclSmem& s = *reinterpret_cast<CclSmem*>(smem_raw);
  const CclGeom geo = ccl_geom(g.H, g.W, g.Wp, blockIdx.x, tiles_x, slice_rows(g), ccl_rows(g));
  const bool rho = phi1 != nullptr;
  const int nruns = ccl_tile_label(s, mask, phi1, geo, conn, status);
  if (nruns < 0) return;
  int32_t* state = sc.tpar + (size_t)blockIdx.x * sc.tile_cap;
  ccl_publish(s, nruns, geo, sc.G, rho, g.H * g.W,
              rho ? state + sc.tile_cap / 2 : tile_list(sc, blockIdx.x));
  if (rho) rz_tile_save(s, nruns, state);
  else ccl_tile_save(s, nruns, state);
}

// glen: entries of G (H*W for labels, 2*H*W for rho keys).
__global__ void k_ccl_merge(const uint32_t* mask, MaskGeom g, int tiles_x, int conn, int32_t* G,
                            int glen, int32_t* status) {
  grid_wait();
  const int Hs = slice_rows(g);
  const int n = merge_units(g.H, g.Wp, tiles_x, Hs, ccl_rows(g));
  const int wpb = blockDim.x >> 5;
  for (int u = blockIdx.x * wpb + (threadIdx.x >> 5); u < n; u += gridDim.x * wpb)
    ccl_merge_unit(mask, g.H, g.W, g.Wp, u, conn, G, glen, status, Hs, ccl_rows(g));
}

__global__ void __launch_bounds__(EXEC_THREADS, 2)
k_ccl_final_labels(const uint32_t* mask, MaskGeom g, int tiles_x, int conn, CclScratch sc,
                   int32_t* status) {
  grid_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CclSmem& s = *reinterpret_cast<CclSmem*>(smem_raw);
  const CclGeom geo = ccl_geom(g.H, g.W, g.Wp, blockIdx.x, tiles_x, slice_rows(g), ccl_rows(g));
  const int nruns = ccl_tile_load(s, mask, geo, conn, sc.tpar + (size_t)blockIdx.x * sc.tile_cap,
                                  tile_list(sc, blockIdx.x), sc.tile_cap, sc.G, g.H * g.W, status);
  if (nruns >= 0) ccl_write_labels(s, nruns, geo, sc.G);
}

__global__ void __launch_bounds__(EXEC_THREADS, 3)
k_rz_final(const uint32_t* phi2, MaskGeom g, int tiles_x, int conn, CclScratch sc, uint32_t* Z,
           int32_t* status) {
  grid_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const CclGeom geo = ccl_geom(g.H, g.W, g.Wp, blockIdx.x, tiles_x, slice_rows(g), ccl_rows(g));
  rz_tile_select(*reinterpret_cast<RzSmem*>(smem_raw), phi2, geo, conn,
                 sc.tpar + (size_t)blockIdx.x * sc.tile_cap, sc.tile_cap, sc.G, g.H * g.W, Z, status);
}

// ----------------------------------------------------------- conversion --

__global__ void k_pack_u8(const uint8_t* src, MaskGeom g, uint32_t* out) {
  const int lane = threadIdx.x & 31;
  const long long nwords = (long long)g.H * g.Wp;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < nwords;
       i += nwarps) {
    int y, w;
    split_index(i, g.Wp, y, w);
    const int x = 32 * w + lane;
    const bool p = (x < g.W) && src[(size_t)y * g.W + x] != 0;
    const uint32_t word = __ballot_sync(FULL, p);
    if (lane == 0) out[i] = word;
  }
}

__global__ void k_unpack_u8(const uint32_t* src, MaskGeom g, uint8_t* out) {
  const long long n = (long long)g.H * g.W;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    int y, x;
    split_index(i, g.W, y, x);
    out[i] = (uint8_t)((__ldg(src + (size_t)y * g.Wp + (x >> 5)) >> (x & 31)) & 1u);
  }
}

// n vectors from src to dst.
constexpr int COPY_UNR = 4;
__global__ void __launch_bounds__(kThreads) k_copy(const uint4* src, uint4* dst,
                                                   unsigned n) {
  grid_wait();
  const unsigned first = blockIdx.x * (kThreads * COPY_UNR) + threadIdx.x;
  uint4 v[COPY_UNR];
#pragma unroll
  for (int u = 0; u < COPY_UNR; ++u)
    if (first + u * kThreads < n) v[u] = __ldcg(src + first + u * kThreads);
#pragma unroll
  for (int u = 0; u < COPY_UNR; ++u)
    if (first + u * kThreads < n) dst[first + u * kThreads] = v[u];
}

__global__ void k_clear_padding(uint32_t* m, MaskGeom g) {
  const long long nwords = (long long)g.H * g.Wp;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nwords;
       i += (long long)gridDim.x * blockDim.x) {
    int y, w;
    split_index(i, g.Wp, y, w);
    m[i] &= vmask(w, g.W);
  }
}

}  // namespace

// ============================================================ wrappers ==

cudaError_t launch_thresholds(const void* plane, int format, MaskGeom g, const ThrSet& T, int n,
                              cudaStream_t st) {
  const int grid = grid_for((long long)g.H * g.Wp * 2, kThreads, 152 * 8);
  switch (n) {
    case 1: return launch_early(k_thresholds<1>, grid, kThreads, 0, st, plane, format, g, T);
    case 2: return launch_early(k_thresholds<2>, grid, kThreads, 0, st, plane, format, g, T);
    case 3: return launch_early(k_thresholds<3>, grid, kThreads, 0, st, plane, format, g, T);
    case THR_SET: return launch_early(k_thresholds<THR_SET>, grid, kThreads, 0, st, plane, format, g, T);
    default: return cudaErrorInvalidValue;
  }
}

template <int OP>
static cudaError_t pointwise(const uint32_t* a, const uint32_t* b, MaskGeom g, uint32_t* out,
                             cudaStream_t st) {
  return launch_early(k_pointwise<OP>, grid_for((long long)g.H * (g.Wp >> 2), kThreads), kThreads, 0,
                      st, reinterpret_cast<const uint4*>(a), reinterpret_cast<const uint4*>(b), g,
                      reinterpret_cast<uint4*>(out));
}
cudaError_t launch_not(const uint32_t* a, MaskGeom g, uint32_t* out, cudaStream_t st) {
  return pointwise<0>(a, nullptr, g, out, st);
}
cudaError_t launch_and(const uint32_t* a, const uint32_t* b, MaskGeom g, uint32_t* out,
                       cudaStream_t st) {
  return pointwise<1>(a, b, g, out, st);
}
cudaError_t launch_or(const uint32_t* a, const uint32_t* b, MaskGeom g, uint32_t* out,
                      cudaStream_t st) {
  return pointwise<2>(a, b, g, out, st);
}
cudaError_t launch_andnot(const uint32_t* a, const uint32_t* b, MaskGeom g, uint32_t* out,
                          cudaStream_t st) {
  return pointwise<5>(a, b, g, out, st);
}
cudaError_t launch_const(MaskGeom g, bool value, uint32_t* out, cudaStream_t st) {
  return value ? pointwise<4>(nullptr, nullptr, g, out, st) : pointwise<3>(nullptr, nullptr, g, out, st);
}
cudaError_t launch_near(const uint32_t* a, MaskGeom g, int conn, uint32_t* out,
                        cudaStream_t st) {
  return launch_early(k_near, grid_for((long long)g.H * (g.Wp >> 2), kThreads), kThreads, 0, st, a, g,
                      conn, reinterpret_cast<uint4*>(out));
}

size_t select_scratch_bytes(int n) {
  return (size_t)std::min(n, SEL_BATCH) * SEL_HIST * sizeof(uint32_t);
}

cudaError_t launch_selects(const SelJob* jobs, int n, int H, int W, int pitch, void* scratch,
                           cudaStream_t st) {
  for (int at = 0; at < n; at += SEL_BATCH) {
    SelBatch B{};
    const int m = std::min(n - at, SEL_BATCH);
    bool wide = false;
    for (int i = 0; i < m; ++i) {
      B.job[i] = jobs[at + i];
      wide |= B.job[i].format != PX_U16;
    }
    B.state = static_cast<uint32_t*>(scratch);
    B.H = H;
    B.W = W;
    B.pitch = pitch;
    cudaError_t e = cudaMemsetAsync(scratch, 0, select_scratch_bytes(m), st);
    if (e) return e;
    const dim3 grid(select_blocks((int64_t)H * W, m, 2 * 152), m);
    // (16-bit keys: two passes of 12 bits after one that missed)
    for (int pass = 0; pass < (wide ? SEL_PASSES : 3); ++pass) {
      if ((e = launch_early(k_sel_pass, grid, EXEC_THREADS, 0, st, B, pass))) return e;
    }
    if ((e = launch_early(k_sel_finish, m, EXEC_THREADS, 0, st, B))) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_arith(int op, const void* a, int a_format, const void* b, int b_format, float c,
                         float* out, int H, int W, int pitch, cudaStream_t st) {
  return launch_early(k_arith, grid_for((long long)H * W, kThreads), kThreads, 0, st, op, a, a_format, b,
                      b_format, c, out, H, W, pitch);
}

int ccl_tiles_y(int H, int Hs, int cth) {
  if (Hs <= 0) Hs = H;
  return (H / Hs) * ((Hs + cth - 1) / cth);
}
int ccl_tiles_x(int Wp) { return (Wp + CCL_TWW - 1) / CCL_TWW; }
size_t ccl_smem_bytes() { return sizeof(CclSmem); }

// The labelling kernels need more than 48 KB of dynamic shared memory; the
// attribute is set once per device (guarded: host threads may call the
// labelling entry points concurrently, on different devices).
namespace {
constexpr int kMaxDevices = 64;
std::mutex g_attr_mu;
bool g_attr_done[kMaxDevices] = {};
}  // namespace

static cudaError_t ccl_set_attrs();
cudaError_t ccl_configure() { return ccl_set_attrs(); }

static cudaError_t ccl_set_attrs() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_attr_mu);
  if (g_attr_done[dev]) return cudaSuccess;
  const int sm = (int)sizeof(CclSmem);
  if ((e = cudaFuncSetAttribute(k_ccl_local, cudaFuncAttributeMaxDynamicSharedMemorySize, sm)))
    return e;
  if ((e = cudaFuncSetAttribute(k_ccl_final_labels,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, sm)))
    return e;
  if ((e = cudaFuncSetAttribute(k_rz_final, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(RzSmem))))
    return e;
  g_attr_done[dev] = true;
  return cudaSuccess;
}

long long ccl_merge_units(int H, int Wp, int Hs, int cth) {
  if (Hs <= 0) Hs = H;
  return (long long)(H / Hs) * ((Hs + cth - 1) / cth - 1) * Wp +
         (long long)(ccl_tiles_x(Wp) - 1) * ((H + 31) / 32);
}
int ccl_tile_cap_host(int Wp, int cth) { return (cth / 2) * std::min(CCL_TWW, Wp) * 32; }

// Labelling kernels come up early where their tiles are one wave (two blocks
// an SM), and not in a captured graph: with more tiles the early blocks are in
// the way of the waves still to come (8192 x 8192: 395 us early, 387 not), and
// between the nodes of a graph there is less to hide (a chain of 75 selects at
// 2048 x 2048: 2.85 ms early, 2.78 not).  On a stream of its own 3001 x 2777
// labelling takes 49 us early and 51.5 not.
static bool ccl_early(int tiles, cudaStream_t st) {
  if (tiles > 2 * 152) return false;
  cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &s) == cudaSuccess) return s == cudaStreamCaptureStatusNone;
  cudaGetLastError();  // (the legacy stream beside another one's capture; the launch says so)
  return false;
}

cudaError_t launch_ccl_labels(const uint32_t* mask, MaskGeom g, int conn, CclScratch sc,
                              int32_t* status, cudaStream_t st) {
  cudaError_t e = ccl_set_attrs();
  if (e) return e;
  const int ty = ccl_tiles_y(g.H, g.Hs, ccl_rows(g)), tx = ccl_tiles_x(g.Wp);
  const size_t sm = sizeof(CclSmem);
  const bool early = ccl_early(ty * tx, st);
  int32_t* labels = sc.G;
  e = launch_kernel(early, k_ccl_local, ty * tx, EXEC_THREADS, sm, st, mask, nullptr, g, tx, conn, sc, status);
  if (e) return e;
  const long long nm = ccl_merge_units(g.H, g.Wp, g.Hs, ccl_rows(g)) * 32LL;
  if (nm > 0) {
    e = launch_kernel(early, k_ccl_merge, grid_for(nm, kThreads), kThreads, 0, st, mask, g, tx, conn, labels,
                     g.H * g.W, status);
    if (e) return e;
  }
  return launch_kernel(early, k_ccl_final_labels, ty * tx, EXEC_THREADS, sm, st, mask, g, tx, conn, sc, status);
}

cudaError_t launch_rz(const uint32_t* phi1, const uint32_t* phi2, MaskGeom g, int conn,
                      CclScratch sc, uint32_t* Z, int32_t* status, cudaStream_t st) {
  cudaError_t e = ccl_set_attrs();
  if (e) return e;
  const int ty = ccl_tiles_y(g.H, g.Hs, ccl_rows(g)), tx = ccl_tiles_x(g.Wp);
  const size_t sm = sizeof(CclSmem);
  const bool early = ccl_early(ty * tx, st);
  e = launch_kernel(early, k_ccl_local, ty * tx, EXEC_THREADS, sm, st, phi2, phi1, g, tx, conn, sc, status);
  if (e) return e;
  const long long nm = ccl_merge_units(g.H, g.Wp, g.Hs, ccl_rows(g)) * 32LL;
  if (nm > 0) {
    e = launch_kernel(early, k_ccl_merge, grid_for(nm, kThreads), kThreads, 0, st, phi2, g, tx, conn, sc.G,
                     2 * g.H * g.W, status);
    if (e) return e;
  }
  return launch_kernel(early, k_rz_final, ty * tx, EXEC_THREADS, sizeof(RzSmem), st, phi2, g, tx, conn, sc, Z,
                      status);
}

cudaError_t launch_pack_u8(const uint8_t* src, MaskGeom g, uint32_t* out, cudaStream_t st) {
  k_pack_u8<<<grid_for((long long)g.H * g.Wp * 32, kThreads * 4), kThreads, 0, st>>>(src, g,
                                                                                    out);
  return cudaGetLastError();
}
cudaError_t launch_unpack_u8(const uint32_t* src, MaskGeom g, uint8_t* out, cudaStream_t st) {
  k_unpack_u8<<<grid_for((long long)g.H * g.W, kThreads * 8), kThreads, 0, st>>>(src, g, out);
  return cudaGetLastError();
}
cudaError_t launch_copy(const void* src, void* dst, size_t bytes, cudaStream_t st) {
  const size_t n = bytes / 16, per_block = (size_t)kThreads * COPY_UNR;
  if (bytes % 16 || n > 0x7FFFFFFFu) return cudaErrorInvalidValue;
  if (!n) return cudaSuccess;
  return launch_early(k_copy, dim3((unsigned)((n + per_block - 1) / per_block)), kThreads, 0, st,
                      static_cast<const uint4*>(src), static_cast<uint4*>(dst), (unsigned)n);
}
cudaError_t launch_clear_padding(uint32_t* m, MaskGeom g, cudaStream_t st) {
  k_clear_padding<<<grid_for((long long)g.H * g.Wp, kThreads * 4), kThreads, 0, st>>>(m, g);
  return cudaGetLastError();
}

}  // namespace vl
