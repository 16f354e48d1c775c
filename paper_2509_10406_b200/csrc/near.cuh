// What the two near-field kernels (stand-in keys of the two-level retrieval) share.
#pragma once
#include "common.cuh"

namespace muse {

constexpr int kNbPairs = 2048, kNbGroup = 8;                // (query, slot) pairs of a chunk at most; earlier blocks per product

__device__ __forceinline__ void nb_mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void nb_cp_async16(void* smem_dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)), "l"(src) : "memory");
}
// counts -> exclusive prefix sums, in place, by one warp
__device__ __forceinline__ void nb_scan(int* off, int n, int lane) {
  int at = 0;
  for (int j0 = 0; j0 < n; j0 += 32) {
    const int cnt = j0 + lane < n ? off[j0 + lane] : 0;
    int pre = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, pre, o); if (lane >= o) pre += v; }
    if (j0 + lane < n) off[j0 + lane] = at + pre - cnt;
    at += __shfl_sync(0xffffffffu, pre, 31);
  }
}

}  // namespace muse
