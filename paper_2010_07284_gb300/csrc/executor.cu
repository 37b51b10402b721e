// Persistent batched executor.
//
// One launch walks a device work list.  An item is a range of sub-items
// (tiles, merge chunks, selects) of one step of one job; items are ordered
// so that everything an item depends on comes earlier in the list.  CTAs pop
// items with an atomic counter, so an item's dependencies were popped by
// CTAs already running: the earliest unfinished item can always progress,
// and the launch needs no co-residency guarantee.  Before running, an item
// waits (bounded, with back-off) until every sub-item of each step its
// step depends on is done; a wait that runs out records VL_ERR_TIMEOUT in the job's
// status word and the job's remaining items are skipped.  This replaces the
// paper's host-side event chaining and host-checked CCL termination
// (Sec. 3.2-3.3) with device-side counters: the host never waits.
#include <cstddef>

#include "dev_ccl.cuh"
#include "dev_common.cuh"
#include "dev_group.cuh"
#include "dev_select.cuh"
#include "kernels.h"

namespace vl {

namespace {

VL_DEV unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

VL_DEV int ld_acquire(const int32_t* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Polls *ctr with back-off until it is at least `need`; false when
// the limit runs out first (a negative one does at once).
VL_DEV bool poll_count(const int32_t* ctr, int need, long long spin_limit, const int32_t* status) {
  long long spins = 0;
  unsigned ns = 32;
  if (spin_limit < 0) return false;
  while (ld_acquire(ctr) < need) {
    if (++spins > spin_limit || (status && ldcg(status) != 0)) return false;
    __nanosleep(ns);
    if (ns < 1024) ns <<= 1;
  }
  return true;
}

// Rank codes of rows [y0, y1) of one channel against the sorted table tv
// (see RankTab): one warp per 32-pixel word, one lane per pixel; code bit b
// of the word's pixels is a ballot, written to plane b (lane b writes it).
// A warp takes RANK_UNR words at a time: their loads are in flight
// together, and their searches (branch-free, the same number of steps for
// every lane) interleave.
constexpr int RANK_UNR = 4;
VL_DEV void rank_rows(const float* tv, const RankTab& T, const void* plane, int format, bool nc,
                      int H, int W, int Wp, int pitch, int y0, int y1, uint32_t* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const size_t pstride = (size_t)H * Wp;
  const int nwords = (y1 - y0) * Wp;
  for (int base = warp * RANK_UNR; base < nwords; base += nw * RANK_UNR) {
    float v[RANK_UNR];
    bool in[RANK_UNR];
#pragma unroll
    for (int u = 0; u < RANK_UNR; ++u) {
      const int idx = base + u;
      const int y = y0 + idx / Wp, w = idx - (idx / Wp) * Wp;
      const int x = 32 * w + lane;
      in[u] = idx < nwords && x < W;
      v[u] = 0.f;
      if (in[u]) {
        const size_t i = (size_t)y * pitch + x;
        if (format == PX_U16) v[u] = (float)static_cast<const unsigned short*>(plane)[i];
        else v[u] = nc ? __ldg(static_cast<const float*>(plane) + i) : __ldcg(static_cast<const float*>(plane) + i);
      }
    }
    // lower bound: the number of table values below v (none for NaN)
    int lo[RANK_UNR];
#pragma unroll
    for (int u = 0; u < RANK_UNR; ++u) lo[u] = 0;
    for (int n = T.m; n > 1;) {
      const int half = n >> 1;
#pragma unroll
      for (int u = 0; u < RANK_UNR; ++u) lo[u] = tv[lo[u] + half - 1] < v[u] ? lo[u] + half : lo[u];
      n -= half;
    }
#pragma unroll
    for (int u = 0; u < RANK_UNR; ++u) {
      const int idx = base + u;
      if (idx >= nwords) break;  // uniform: idx is the same for the warp
      if (T.m > 0 && tv[lo[u]] < v[u]) ++lo[u];
      const unsigned code = 2u * (unsigned)lo[u] + ((lo[u] < T.m && tv[lo[u]] == v[u]) ? 1u : 0u);
      uint32_t mine = 0;
      for (int b = 0; b < T.nbits; ++b) {
        const uint32_t word = __ballot_sync(FULL, in[u] && ((code >> b) & 1u));
        if (lane == b) mine = word;
      }
      const uint32_t nan = __ballot_sync(FULL, in[u] && v[u] != v[u]);
      if (lane == T.nbits) mine = nan;
      const int y = y0 + idx / Wp, w = idx - (idx / Wp) * Wp;
      if (lane <= T.nbits) out[(size_t)lane * pstride + (size_t)y * Wp + w] = mine;
    }
  }
}

// One operation, rounded once: the _rn intrinsics are never contracted into
// fused multiply-adds.
VL_DEV float arith_op(uint32_t op, float u, float w) {
  switch (op) {
    case A_ADD: return __fadd_rn(u, w);
    case A_SUB: return __fsub_rn(u, w);
    case A_MUL: return __fmul_rn(u, w);
    default: return __fdiv_rn(u, w);
  }
}

// Number terms of rows [sub * ARITH_ROWS, +ARITH_ROWS), for VECS vectors of
// four pixels a thread at a time: instructions, with the images' addresses in
// them, and the registers (q of vector u of thread t at R[(q * VECS + u) * nt +
// t]) lie in shared memory; nt threads work.  Pixels behind a row's end are worked
// out too: rows are 32 * Wp elements long.
//
// Bound by latency, of the loads and of one instruction after the other, so
// as many vectors as the registers leave room for, and four rows an item, so
// that an image of a thousand rows has items for most blocks.  (Nine
// instructions on two 1021 x 1530 uint16 channels: 11.6 us; pixel by pixel, in
// items of eight rows, 54.)
constexpr int ARITH_PROG_BYTES = 16 * kArithMaxInsns;
template <int VECS>
VL_DEV void arith_rows(const DevJob& J, int sub, unsigned char* smem, int nt) {
  const int n = J.n_arith;
  uint4* prog = reinterpret_cast<uint4*>(smem);
  float4* r = reinterpret_cast<float4*>(smem + ARITH_PROG_BYTES) + threadIdx.x;
  const size_t plane = (size_t)J.H * J.pitch;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const ArithInsn A = J.arith[i];
    uint4 w = make_uint4(A.op | A.dst << 8 | A.a << 16 | (uint32_t)A.b << 24, __float_as_uint(A.c), 0u, 0u);
    if (A.op == A_VALUE || A.op == A_STORE) {
      const DevImage im = J.images[A.op == A_VALUE ? A.img : J.first_num_image + A.img];
      const unsigned long long p = (unsigned long long)chan_ptr(im, A.op == A_VALUE ? A.ch : 0, plane);
      w.y = (im.format == PX_U16 ? 1u : 0u) | (im.written ? 2u : 0u);
      w.z = (uint32_t)p;
      w.w = (uint32_t)(p >> 32);
    }
    prog[i] = w;
  }
  __syncthreads();
  const int y0 = sub * ARITH_ROWS, rows = min(J.H - y0, ARITH_ROWS), vpr = (J.W + 3) >> 2;
  const int total = rows * vpr;
  if ((int)threadIdx.x >= nt) return;
  for (int first = threadIdx.x; first < total; first += nt * VECS) {
    size_t off[VECS];
#pragma unroll
    for (int u = 0; u < VECS; ++u) {
      const int idx = min(first + u * nt, total - 1);  // (the last vector again: the same values)
      const int y = idx / vpr;
      off[u] = (size_t)(y0 + y) * J.pitch + 4 * (idx - y * vpr);
    }
    for (int k = 0; k < n; ++k) {
      const uint4 A = prog[k];
      const uint32_t op = A.x & 0xFFu, dst = (A.x >> 8) & 0xFFu, a = (A.x >> 16) & 0xFFu, b = A.x >> 24;
      void* p = reinterpret_cast<void*>((unsigned long long)A.z | (unsigned long long)A.w << 32);
      if (op == A_VALUE) {
        float4 v[VECS];
#pragma unroll
        for (int u = 0; u < VECS; ++u) v[u] = ld_px4(p, A.y & 1u ? PX_U16 : PX_F32, !(A.y & 2u), off[u]);
#pragma unroll
        for (int u = 0; u < VECS; ++u) r[(dst * VECS + u) * nt] = v[u];
      } else if (op == A_STORE) {
#pragma unroll
        for (int u = 0; u < VECS; ++u)
          *reinterpret_cast<float4*>(static_cast<float*>(p) + off[u]) = r[(a * VECS + u) * nt];
      } else {
        const float c = __uint_as_float(A.y);
#pragma unroll
        for (int u = 0; u < VECS; ++u) {
          const float4 x = r[(a * VECS + u) * nt];
          const float4 y = b == kArithConst ? make_float4(c, c, c, c) : r[(b * VECS + u) * nt];
          r[(dst * VECS + u) * nt] = make_float4(arith_op(op, x.x, y.x), arith_op(op, x.y, y.y),
                                                 arith_op(op, x.z, y.z), arith_op(op, x.w, y.w));
        }
      }
    }
  }
}

// The executor's dynamic shared memory, by name: through a pointer argument
// its accesses would be generic ones.
extern __shared__ __align__(16) unsigned char exec_smem[];
// The job and the step of the item at hand (read by every sub-item; from
// global memory each of their fields is a dependent access of its own).
__shared__ DevJob s_job;
__shared__ StepDesc s_step;
static_assert(sizeof(DevJob) % 8 == 0 && sizeof(StepDesc) <= 128, "copied by one warp");

// The kinds of sub-items, each a function of its own: the registers of one
// then do not depend on what the others keep alive (inlined into one kernel
// at 64 registers a thread, the interpreter's loop spilled).

VL_DEV SelChan select_chan(const DevJob& J, const PctDesc& d) {
  const DevImage im = J.images[d.img];
  return SelChan{chan_ptr(im, d.ch, (size_t)J.H * J.pitch), im.format, !im.written, J.H, J.W, J.pitch};
}
VL_DEV long long select_rank_of(const DevJob& J, const PctDesc& d) {
  return (long long)(d.q * (double)((long long)J.H * J.W - 1));
}
__device__ __noinline__ void percentile_item(int sub, int smem_bytes) {
  const DevJob& J = s_job;
  SelectSmem& s = *reinterpret_cast<SelectSmem*>(exec_smem);
  const PctDesc d = J.pct[s_step.pct_off + sub];
  const SelChan c = select_chan(J, d);
  const float v =
      J.sel_hist ? sel_finish(s, J.sel_hist + (size_t)sub * SEL_HIST, c, select_rank_of(J, d))
                 : select_rank(s, reinterpret_cast<uint32_t*>(exec_smem + sizeof(SelectSmem)),
                               (smem_bytes - (int)sizeof(SelectSmem)) / 4, c, select_rank_of(J, d), J.status);
  if (threadIdx.x == 0) J.pct_val[d.slot] = v;
}
__device__ __noinline__ void percentile_pass_item(int sub) {
  const DevJob& J = s_job;
  const int k = sub / J.sel_blocks, block = sub - k * J.sel_blocks;
  const PctDesc d = J.pct[s_step.pct_off + k];
  sel_pass(*reinterpret_cast<SelectSmem*>(exec_smem), select_chan(J, d), s_step.halo, block,
           J.sel_blocks, select_rank_of(J, d), J.sel_hist + (size_t)k * SEL_HIST);
}

__device__ __noinline__ void group_item(int sub, const ExecLaunch& L) {
  const DevJob& J = s_job;
  const StepDesc& S = s_step;
  group_tile(J, S, sub, reinterpret_cast<uint32_t*>(exec_smem), L.smem_bytes / 4, L.group_buffers);
}

__device__ __noinline__ void rank_item(int sub) {
  const DevJob& J = s_job;
  const int per_tab = (J.H + RANK_ROWS - 1) / RANK_ROWS;
  const int tab = sub / per_tab, rb = sub - tab * per_tab;
  const RankTab T = J.rtab[tab];
  float* tv = reinterpret_cast<float*>(exec_smem);
  for (int i = threadIdx.x; i < T.m; i += blockDim.x) tv[i] = J.rvals[T.val_off + i];
  __syncthreads();
  const DevImage im = J.images[T.img];
  rank_rows(tv, T, chan_ptr(im, T.ch, (size_t)J.H * J.pitch), im.format, !im.written, J.H,
            J.W, J.Wp, J.pitch, rb * RANK_ROWS, min(J.H, (rb + 1) * RANK_ROWS),
            J.planes + (size_t)T.plane0 * J.H * J.Wp);
}

__device__ __noinline__ void arith_item(int sub, int smem_bytes) {
  const int reg = 16 * EXEC_THREADS;  // bytes of a register, a vector each thread
  const int room = (smem_bytes - ARITH_PROG_BYTES) / (reg * max(s_job.arith_regs, 1));
  if (room >= 4) arith_rows<4>(s_job, sub, exec_smem, EXEC_THREADS);
  else if (room >= 2) arith_rows<2>(s_job, sub, exec_smem, EXEC_THREADS);
  else arith_rows<1>(s_job, sub, exec_smem, room ? EXEC_THREADS : EXEC_THREADS / 2);
}

__device__ __noinline__ void rz_local_item(int sub, int per_rz) {
  const DevJob& J = s_job;
  const StepDesc& S = s_step;
  const int npx = J.H * J.W;
  CclSmem& s = *reinterpret_cast<CclSmem*>(exec_smem);
  const int j = sub / per_rz, tile = sub - j * per_rz;
  const RzDesc r = J.rz[S.rz_off + j];
  const int k = r.scratch;
  const CclGeom geo = ccl_geom(J.H, J.W, J.Wp, tile, J.c_tiles_x, J.H, J.c_th);
  const int nruns = ccl_tile_label(s, slot_ptr(J, r.phi2_slot), slot_ptr(J, r.phi1_slot), geo, J.conn,
                                   J.status);
  if (nruns < 0) return;
  int32_t* state = rz_state(J, k) + (size_t)tile * J.tile_cap;
  ccl_publish(s, nruns, geo, rz_G(J, k), true, npx, state + J.tile_cap / 2);
  rz_tile_save(s, nruns, state);
}

__device__ __noinline__ void rz_final_item(int sub, int per_rz) {
  const DevJob& J = s_job;
  const StepDesc& S = s_step;
  const int npx = J.H * J.W;
  const int j = sub / per_rz, tile = sub - j * per_rz;
  const RzDesc r = J.rz[S.rz_off + j];
  const int k = r.scratch;
  const CclGeom geo = ccl_geom(J.H, J.W, J.Wp, tile, J.c_tiles_x, J.H, J.c_th);
  rz_tile_select(*reinterpret_cast<RzSmem*>(exec_smem), slot_ptr(J, r.phi2_slot), geo, J.conn,
                 rz_state(J, k) + (size_t)tile * J.tile_cap, J.tile_cap, rz_G(J, k), npx,
                 slot_ptr(J, r.z_slot), J.status);
}

__device__ __noinline__ void rz_merge_item(int sub, int per_rz) {
  const DevJob& J = s_job;
  const StepDesc& S = s_step;
  const int npx = J.H * J.W;
  const int j = sub / per_rz, chunk = sub - j * per_rz;
  const RzDesc r = J.rz[S.rz_off + j];
  const uint32_t* phi2 = slot_ptr(J, r.phi2_slot);
  const int n = merge_units(J.H, J.Wp, J.c_tiles_x, J.H, J.c_th);
  const int nw = blockDim.x >> 5;
  for (int u = chunk * nw + (threadIdx.x >> 5); u < n; u += per_rz * nw)
    ccl_merge_unit(phi2, J.H, J.W, J.Wp, u, J.conn, rz_G(J, r.scratch),
                   2 * npx, J.status, J.H, J.c_th);
}

VL_DEV void run_subitem(int sub, int per_rz, const ExecLaunch& L) {
  switch (s_step.kind) {
    case SK_PCT: percentile_item(sub, L.smem_bytes); break;
    case SK_PCT_PASS: percentile_pass_item(sub); break;
    case SK_GROUP: group_item(sub, L); break;
    case SK_RANK: rank_item(sub); break;
    case SK_ARITH: arith_item(sub, L.smem_bytes); break;
    case SK_RZ_LOCAL: rz_local_item(sub, per_rz); break;
    case SK_RZ_MERGE: rz_merge_item(sub, per_rz); break;
    case SK_RZ_FINAL: rz_final_item(sub, per_rz); break;
    default: break;
  }
}

// What an item costs besides its work is a chain of round trips to L2, about
// 0.4 us each: the pop, the item, its job and step together (StepRec), and
// the counters it waits for, all at once by a lane each.  The next item is
// popped before the fence behind the finished one, so that the two wait
// together; a popped item never waits for another one of its own block, so
// the earliest unfinished item still always progresses.  (With the
// fields read one from the other, waits one after the other and a fence by
// every thread, 2000 nodes at 2048 x 2048 took 5.26 ms instead of 4.94, 1024
// slices 5.07 instead of 4.66.)
__global__ void __launch_bounds__(EXEC_THREADS, 2) k_exec(const __grid_constant__ ExecLaunch L) {
  __shared__ WorkItem s_item;
  __shared__ int s_go;  // -1: no more items, 0: skip, 1: run
  __shared__ int s_per_rz;
  int next = 0;         // (thread 0) the item popped last
  if (threadIdx.x == 0) next = atomicAdd(L.head, 1);
  for (;;) {
    unsigned long long t_pop = 0, t_go = 0;
    if (threadIdx.x < 32) {
      // warp 0 brings the item's job and step to shared memory and waits for
      // the steps the item depends on
      const int lane = threadIdx.x;
      const int idx = __shfl_sync(FULL, next, 0);
      if (idx >= L.n_items) {
        if (lane == 0) s_go = -1;
      } else {
        const WorkItem it = L.items[idx];
        const int rec = __ldg(reinterpret_cast<const int*>(L.steps + it.step) + lane);
        const unsigned long long* src = reinterpret_cast<const unsigned long long*>(L.jobs + it.job);
        for (int k = lane; k < (int)(sizeof(DevJob) / 8); k += 32)
          reinterpret_cast<unsigned long long*>(&s_job)[k] = __ldg(src + k);
        constexpr int STEP = sizeof(StepDesc) / 4, DEP = offsetof(StepRec, dep) / 4;
        if (lane < STEP) reinterpret_cast<int*>(&s_step)[lane] = rec;
        if (lane == offsetof(StepRec, per_rz) / 4) s_per_rz = rec;
        if (L.trace && lane == 0) t_pop = now_ns();
        const int n_deps = __shfl_sync(FULL, rec, offsetof(StepRec, n_deps) / 4);
        const int more = __shfl_sync(FULL, rec, offsetof(StepRec, more) / 4);
        const int dep = __shfl_sync(FULL, rec, DEP + 2 * (lane & (REC_DEPS - 1)));
        const int need = __shfl_sync(FULL, rec, DEP + 2 * (lane & (REC_DEPS - 1)) + 1);
        // (a negative limit makes every wait expire at once: tests of the
        // timeout path)
        bool ok = true;
        if (lane < min(n_deps, REC_DEPS)) ok = poll_count(L.done + dep, need, L.spin_limit, nullptr);
        for (int q = REC_DEPS + lane; q < n_deps && ok; q += 32) {
          const StepRec::Dep d = L.more_deps[more + q - REC_DEPS];
          ok = poll_count(L.done + d.step, d.need, L.spin_limit, nullptr);
        }
        ok = __all_sync(FULL, ok);
        __syncwarp();  // (the status is read after every lane's wait)
        if (lane == 0) {
          s_item = it;
          if (!ok) set_status(s_job.status, ST_TIMEOUT);
          s_go = ok && ldcg(s_job.status) == 0;
          if (L.trace) t_go = now_ns();
        }
      }
    }
    __syncthreads();
    if (s_go < 0) break;
    const WorkItem it = s_item;
    if (s_go) {
      const int per_rz = s_per_rz;
      for (int k = 0; k < it.count; ++k) {
        run_subitem(it.first + k, per_rz, L);
        __syncthreads();
      }
    } else {
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      // the block's writes come before its count: the barrier above orders
      // them before this thread's fence, and the fence before the count
      next = atomicAdd(L.head, 1);
      __threadfence();
      atomicAdd(L.done + it.step, it.count);
      if (L.trace) {
        const unsigned long long t_end = now_ns();
        unsigned long long* tr = L.trace + 4 * (size_t)it.step;
        atomicMin(tr + 0, t_go);
        atomicMax(tr + 1, t_end);
        atomicAdd(tr + 2, t_end - t_go);
        atomicAdd(tr + 3, t_go - t_pop);
      }
    }
  }
}

}  // namespace

size_t exec_smem_bytes(int group_buffers, int group_rows, int tile_words) {
  size_t g = GROUP_PROG_BYTES + (size_t)group_buffers * group_buffer_bytes(group_rows, tile_words);
  size_t m = sizeof(CclSmem);
  if (sizeof(SelectSmem) > m) m = sizeof(SelectSmem);
  const size_t arith = (size_t)kArithMaxRegs * (EXEC_THREADS / 2) * 16 + ARITH_PROG_BYTES;
  if (arith > m) m = arith;
  if (g > m) m = g;
  return (m + 15) & ~(size_t)15;
}

cudaError_t exec_configure(size_t smem_bytes, int* max_ctas_per_sm) {
  cudaError_t e = cudaFuncSetAttribute(k_exec, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem_bytes);
  if (e) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(max_ctas_per_sm, k_exec, EXEC_THREADS,
                                                       smem_bytes);
}

cudaError_t launch_exec(const ExecLaunch& L, cudaStream_t st) {
  k_exec<<<L.grid, EXEC_THREADS, (size_t)L.smem_bytes, st>>>(L);
  return cudaGetLastError();
}

}  // namespace vl
