// Tensor memory (TMEM, 256 KB per SM as 128 lanes x 512 columns of 32 bits) as a per-thread
// store: warp w of a block owns lanes 32 (w mod 4) .. + 31, and a thread reads and writes runs of
// 8 columns of its own lane.  Nothing here is a matrix operand; the column pass keeps values
// there that each thread reads back itself (the reference field and the residual sum of its
// crop rows, its chirp entries), so they take neither registers nor shared memory.
//
// A block allocates a power of two of columns (>= 32) once and frees them before it ends.  An
// allocation waits in hardware until the SM has that many columns free: the grids are sized so
// that the resident blocks' columns fit, and a block of another kernel holds its columns only
// until it ends.

#pragma once

#include <cstdint>

#include "holo_tma.cuh"

namespace holo {

__host__ __device__ constexpr int tmem_pow2(int c) {
  int p = 32;
  while (p < c) p *= 2;
  return p;
}

// One warp of the block; the address lands in *dst (shared memory, read after a barrier).
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, int columns) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_addr(dst)),
               "r"(columns)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t base, int columns) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(columns)
               : "memory");
}
// The calling thread's lane run: `words` columns per thread, warps 4 apart side by side.
__device__ __forceinline__ uint32_t tmem_own(uint32_t base, int words) {
  const uint32_t w = threadIdx.x >> 5;
  return base + ((w & 3u) << 21) + (w >> 2) * (uint32_t)words;
}

// 4 complex values (8 columns) of the calling thread's lane; every lane of the warp takes part.
__device__ __forceinline__ void tmem_load4(float2 (&x)[4], uint32_t addr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(x[0].x), "=f"(x[0].y), "=f"(x[1].x), "=f"(x[1].y), "=f"(x[2].x), "=f"(x[2].y),
        "=f"(x[3].x), "=f"(x[3].y)
      : "r"(addr)
      : "memory");
}
// two runs with one wait
__device__ __forceinline__ void tmem_load4x2(float2 (&x)[4], float2 (&y)[4], uint32_t ax,
                                             uint32_t ay) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%16];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8, %9, %10, %11, %12, %13, %14, %15}, [%17];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(x[0].x), "=f"(x[0].y), "=f"(x[1].x), "=f"(x[1].y), "=f"(x[2].x), "=f"(x[2].y),
        "=f"(x[3].x), "=f"(x[3].y), "=f"(y[0].x), "=f"(y[0].y), "=f"(y[1].x), "=f"(y[1].y),
        "=f"(y[2].x), "=f"(y[2].y), "=f"(y[3].x), "=f"(y[3].y)
      : "r"(ax), "r"(ay)
      : "memory");
}
// Stores of one thread become visible to its later loads after tmem_store_done.
__device__ __forceinline__ void tmem_store4(uint32_t addr, const float2 (&x)[4]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"f"(
          x[0].x),
      "f"(x[0].y), "f"(x[1].x), "f"(x[1].y), "f"(x[2].x), "f"(x[2].y), "f"(x[3].x), "f"(x[3].y),
      "r"(addr)
      : "memory");
}
__device__ __forceinline__ void tmem_store_done() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

}  // namespace holo
