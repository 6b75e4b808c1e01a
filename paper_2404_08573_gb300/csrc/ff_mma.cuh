// Warp-level bf16 MMA for the thin or few-row contractions that a 128-row
// tcgen05 tile would leave mostly empty.
#pragma once

#include <cstdint>

namespace ff {

// D (16 x 8, fp32) += A (16 x 16, bf16) B (16 x 8, bf16).  Lane 4 g + t holds
// of A rows g and g + 8 at K slots 2t, 2t+1 (a0, a1) and 2t+8, 2t+9 (a2, a3),
// of B column g at the same slots (b0, b1), of D rows g (d0, d1) and g + 8
// (d2, d3) at columns 2t, 2t+1.
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// A short MMA chain's sums into fp32 registers, rounded to nearest (the
// chain itself is not: the shorter, the less it drifts).
__device__ __forceinline__ void mma_add(float (&d)[4], const float (&t)[4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) d[e] = __fadd_rn(d[e], t[e]);
}

}  // namespace ff
