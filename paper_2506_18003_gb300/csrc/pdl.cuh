// Programmatic dependent launch: a kernel launched by launch_dependent may be set up, and its CTAs
// placed as room becomes free, while the kernel before it on the stream is still running; it touches
// nothing that kernel writes, and writes nothing it reads, before wait_for_previous().  Every kernel
// launched this way calls wait_for_previous() in every CTA, so that kernels still complete in stream order.
// Two rules keep that sound.  A kernel lets the next one start only after its own wait, so that at most two
// kernels of a stream are resident at a time and everything before the earlier one has completed: what a
// kernel reads before its wait (tables, the window of ssca_lag.cuh's channel pass) is written two or more
// kernels back.  And what any kernel of the stream may write is read with load_written(), never with __ldg:
// the read-only path promises correct values only for data that nothing writes while the kernel is resident,
// and here the writer may still be running when the reader's CTAs are placed.
// (Back to back on one stream: a FAM estimate of 280 samples 8.5 -> 5.8 us, two kernels of one and nine
// CTAs; SSCA N = 2^16, Np = 256 82 -> 76 us, three kernels.)
#pragma once
#include <cuda_runtime.h>

namespace scd {

// The next kernel on the stream may be set up once every CTA has called this or ended.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Returns when the kernels before this one have completed and their writes are visible.
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Ordinary (coherent) loads of what an earlier kernel of the stream wrote, after wait_for_previous().
__device__ __forceinline__ float2 load_written(const float2* p) {
  float2 v;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(__cvta_generic_to_global(p)));
  return v;
}
__device__ __forceinline__ float4 load_written(const float4* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(__cvta_generic_to_global(p)));
  return v;
}
__device__ __forceinline__ float load_written(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(__cvta_generic_to_global(p)));
  return v;
}

// early: false launches it the ordinary way, for persistent grids that leave room on the SMs (their CTAs,
// placed while the previous kernel's still take some of it, would pile up on the SMs that empty first).
template <class... P, class... A>
cudaError_t launch_dependent(bool early, void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem,
                             cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1] = {};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace scd
