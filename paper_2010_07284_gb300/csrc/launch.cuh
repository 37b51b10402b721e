// Kernels that follow one another on a stream, each of the next ones coming up
// while the one before still runs (programmatic dependent launch): what a
// kernel of a few microseconds pays for its launch then passes beside its
// predecessor's work.
//
// A kernel launched this way calls grid_wait before it touches memory: by
// every thread, so that a kernel that has ended has waited for all before it,
// and the next one's wait covers those too.  Pointers that are read through the
// read-only path go through grid_wait as well: the compiler may move such
// loads over any barrier that their address does not depend on.
#pragma once
#include "dev_common.cuh"

namespace vl {

VL_DEV void grid_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
VL_DEV void behind_wait() {}
template <class T, class... R>
VL_DEV void behind_wait(T*& p, R&... rest) {
  asm volatile("" : "+l"(p) : : "memory");
  behind_wait(rest...);
}
template <class T, class... R>
VL_DEV void grid_wait(T*& p, R&... rest) {
  grid_wait();
  behind_wait(p, rest...);
}

// early = false: the kernel waits for the one before to end, as usual.
template <class... P, class... A>
cudaError_t launch_kernel(bool early_start, void (*kernel)(P...), dim3 grid, int threads, size_t smem,
                          cudaStream_t st, A... args) {
  cudaLaunchAttribute early{};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &early;
  cfg.numAttrs = early_start ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <class... P, class... A>
cudaError_t launch_early(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st,
                         A... args) {
  return launch_kernel(true, kernel, grid, threads, smem, st, args...);
}

}  // namespace vl
