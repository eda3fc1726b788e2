// Tensor memory (TMEM, 128 lanes x 512 columns of 32 bits per SM) as storage for per-thread FP32
// accumulators: sums that every thread reads and writes at its own points only, once per convolution,
// and that neither the register file nor shared memory has room for.  Warp w of a block reaches lanes
// [32 (w mod 4), 32 (w mod 4) + 32), so the four warps of a warpgroup share a column range and each
// thread owns one lane of it: WORDS columns per warpgroup give every thread WORDS private words.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace qbe {

// Columns to allocate for NT threads with WORDS words each (a power of two, at least 32).
__host__ __device__ constexpr int tmem_columns(int nt, int words) {
  const int need = (nt + 127) / 128 * words;
  int c = 32;
  while (c < need) c *= 2;
  return c;
}

// Allocation by warp 0 (the address goes through shared memory), ending with a block barrier.  One
// block (or two with half the columns each) fits an SM beside its shared memory, so the columns are
// free when it starts; a block frees its own with tmem_free before it ends.
template <int COLS>
__device__ __forceinline__ uint32_t tmem_alloc(uint32_t* slot) {
  if (threadIdx.x < 32) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(slot);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s), "n"(COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return *slot;
}
template <int COLS>
__device__ __forceinline__ void tmem_free(uint32_t base) {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "n"(COLS) : "memory");
  }
}
// The calling thread's WORDS words (address of the first).
template <int WORDS>
__device__ __forceinline__ uint32_t tmem_mine(uint32_t base) {
  const uint32_t w = threadIdx.x >> 5;
  return base + ((32u * (w & 3u)) << 16) + (w >> 2) * WORDS;
}

// Loads are complete after tmem_wait_ld, stores after tmem_wait_st.  All are warp-collective.
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld4(uint32_t a, float* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
               : "r"(a));
}
__device__ __forceinline__ void tmem_st4(uint32_t a, const float* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v[0]), "f"(v[1]),
               "f"(v[2]), "f"(v[3])
               : "memory");
}
template <int CNT>
__device__ __forceinline__ void tmem_ld(uint32_t a, float (&v)[CNT]) {
  static_assert(CNT % 4 == 0, "whole groups of four columns");
#pragma unroll
  for (int i = 0; i < CNT; i += 4) tmem_ld4(a + i, v + i);
}
// Waits for the thread's loads and ties their destinations to the wait, so that no use of them can be
// scheduled before it.
template <int CNT>
__device__ __forceinline__ void tmem_wait_ld(float (&v)[CNT]) {
  tmem_wait_ld();
#pragma unroll
  for (int i = 0; i < CNT; ++i) asm volatile("" : "+f"(v[i]));
}
template <int CNT>
__device__ __forceinline__ void tmem_st(uint32_t a, const float (&v)[CNT]) {
#pragma unroll
  for (int i = 0; i < CNT; i += 4) tmem_st4(a + i, v + i);
}

__device__ __forceinline__ float quad_at(const float4& q, int i) { return i == 0 ? q.x : i == 1 ? q.y : i == 2 ? q.z : q.w; }
// Adds four floats in memory (16-byte aligned), nothing returned.
__device__ __forceinline__ void red_add4(float4* p, float a, float b, float c, float d) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d)
               : "memory");
}

// Eight consecutive columns from / to registers named one by one.
__device__ __forceinline__ void tmem_ld8(uint32_t a, float& v0, float& v1, float& v2, float& v3, float& v4, float& v5,
                                         float& v6, float& v7) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(v0), "=f"(v1), "=f"(v2), "=f"(v3), "=f"(v4), "=f"(v5), "=f"(v6), "=f"(v7)
               : "r"(a));
}
__device__ __forceinline__ void tmem_st8(uint32_t a, float v0, float v1, float v2, float v3, float v4, float v5,
                                         float v6, float v7) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(a), "f"(v0),
               "f"(v1), "f"(v2), "f"(v3), "f"(v4), "f"(v5), "f"(v6), "f"(v7)
               : "memory");
}
// Complex values: real parts in columns a .. a + CNT, imaginary parts in b .. b + CNT (CNT a multiple
// of 8); element i of the columns is v[i * STRIDE].
template <int CNT, int STRIDE = 1>
__device__ __forceinline__ void tmem_ld_c(uint32_t a, uint32_t b, float2* v) {
#pragma unroll
  for (int i = 0; i < CNT; i += 8) {
    float2* p = v + i * STRIDE;
    constexpr int S = STRIDE;
    tmem_ld8(a + i, p[0].x, p[S].x, p[2 * S].x, p[3 * S].x, p[4 * S].x, p[5 * S].x, p[6 * S].x, p[7 * S].x);
    tmem_ld8(b + i, p[0].y, p[S].y, p[2 * S].y, p[3 * S].y, p[4 * S].y, p[5 * S].y, p[6 * S].y, p[7 * S].y);
  }
}
template <int CNT, int STRIDE = 1>
__device__ __forceinline__ void tmem_st_c(uint32_t a, uint32_t b, const float2* v) {
#pragma unroll
  for (int i = 0; i < CNT; i += 8) {
    const float2* p = v + i * STRIDE;
    constexpr int S = STRIDE;
    tmem_st8(a + i, p[0].x, p[S].x, p[2 * S].x, p[3 * S].x, p[4 * S].x, p[5 * S].x, p[6 * S].x, p[7 * S].x);
    tmem_st8(b + i, p[0].y, p[S].y, p[2 * S].y, p[3 * S].y, p[4 * S].y, p[5 * S].y, p[6 * S].y, p[7 * S].y);
  }
}
// tmem_wait_ld for complex destinations.
template <int CNT>
__device__ __forceinline__ void tmem_wait_ld_c(float2* v) {
  tmem_wait_ld();
#pragma unroll
  for (int i = 0; i < CNT; ++i) asm volatile("" : "+f"(v[i].x), "+f"(v[i].y));
}

}  // namespace qbe
