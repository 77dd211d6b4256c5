// Tensor memory accelerator helpers: tile and bulk loads into shared memory whose completion an
// mbarrier counts (initialised, waited for with a bound and invalidated through umma.cuh), and the host
// side's tensor maps.
#pragma once
#include <cuda.h>

#include "tiles.cuh"

namespace scd {

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_expect_tx(uint64_t* mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(su32(mbar)), "r"(bytes) : "memory");
}

// One box of a 3-D tensor map into shared memory; x is the innermost coordinate (x times the element
// size a multiple of 16 bytes).
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* tm, int x, int y, int z, uint64_t* mbar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      :: "r"(su32(dst)), "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(z), "r"(su32(mbar))
      : "memory");
}

// `bytes` contiguous bytes (all three a multiple of 16) into shared memory.
__device__ __forceinline__ void tma_load_bulk(void* dst, const void* src, uint32_t bytes, uint64_t* mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               :: "r"(su32(dst)), "l"(src), "r"(bytes), "r"(su32(mbar)) : "memory");
}

// this thread's shared-memory accesses before a later TMA write to the same addresses
__device__ __forceinline__ void fence_before_tma() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Tensor map over complex64 values moved as raw 64-bit words (cols_tma.cu): dims innermost first,
// strides in bytes of dimensions 1.. (multiples of 16), base 16-byte aligned.
cudaError_t encode_map_c64(CUtensorMap* tm, const void* base, int rank, const cuuint64_t* dims,
                           const cuuint64_t* strides, const cuuint32_t* box);

}  // namespace scd
