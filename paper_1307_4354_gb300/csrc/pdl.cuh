// Programmatic dependent launch: a kernel launched with launch_pdl may start
// while the kernel before it in the stream drains.  It reads its static inputs
// (tables built with the hierarchy), then calls wait_prior() and only then
// touches what earlier kernels wrote or still read.  Completion has to be
// transitive along the stream: a grid completes only after the one before it if
// at least one of its threads calls wait_prior().  Threads without work return
// before that, so nothing is launched this way over an empty set.
// Values written by earlier kernels are read with ld_prior: a plain (coherent)
// load that the compiler keeps behind the wait, which it need not do for
// __ldg.  A V-cycle is some 80 kernels of 2 to 100 us, each of which otherwise
// starts about 1 us after the one before it has ended.
#pragma once

#include "cpm_internal.cuh"

namespace cpm {

// Let the next kernel of the stream be scheduled as this one's blocks drain.
// Not for the largest grids: there the signal of every block costs more than
// the overlap gives (extension over 78 thousand tiles: 82 us with it, 73 us
// without; a mixed solve of five outer iterations at dx = 1/256 25.3 ms with this
// limit, 25.9 without), and the next kernel follows the last block's end.
constexpr unsigned kReleaseBlocks = 32768;
__device__ __forceinline__ void release_next() {
  if (gridDim.x <= kReleaseBlocks) asm volatile("griddepcontrol.launch_dependents;");
}
// Wait until the kernels before this one are complete and their writes visible.
__device__ __forceinline__ void wait_prior() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ float ld_prior(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double ld_prior(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float2 ld_prior(const float2* p) {
  float2 v;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_prior(const float4* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p)
               : "memory");
  return v;
}

// early: the kernel's blocks may be placed while the kernel before it drains.
// They then go where that one leaves room, unevenly, which costs a kernel of
// about one wave of blocks that is bound by the FP64 pipe more than its start:
// with the 3-D FP64 extension and the FP64 GEMV placed early, FP64 solves took
// 9.6 ms (unit sphere, dx = 1/32), 31.7 ms (1/96), 1.28 ms (circle, 1/64), else
// 5.6, 29.5 and 1.21 ms.  The 3-D FP64 extension in relative form is the same
// kernel (relative-form FP64 solves at dx = 1/32 9.4 ms, else 7.6; a torus at 1/44
// 24.2 and 22.4).  The FP32 extension gains from it (an FP32 V-cycle at dx = 1/128
// 0.56 ms, 0.62 without).
template <typename... P, typename... A>
void launch_dep(bool early, void (*kernel)(P...), unsigned grid, unsigned block, cudaStream_t st, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = early ? 1 : 0;
  CPM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, P(args)...));
}
template <typename... P, typename... A>
void launch_pdl(void (*kernel)(P...), unsigned grid, unsigned block, cudaStream_t st, A... args) {
  launch_dep(true, kernel, grid, block, st, args...);
}

}  // namespace cpm
