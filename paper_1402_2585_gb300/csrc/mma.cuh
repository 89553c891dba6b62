// The 16-bit warp-level matrix instruction of the hop passes (hop_tc.cuh).
#pragma once

#include <type_traits>

#include "common.cuh"

namespace hdcg {
namespace tch {

// d += a b, m16n8k16: fragment rows g, g + 8 (g = lane / 4), k 2 t, 2 t + 1 and
// 2 t + 8, 2 t + 9 (t = lane % 4), column g of b, columns 2 t, 2 t + 1 of d; exact
// 16-bit products.  The FP32 sum is truncated towards zero: to 1 it adds nothing of
// 3/4 ulp and 1 of 7/4 ulp, measured.  Long sums of one sign drift (512 products
// summed in one accumulator: 2.6e-6), so contractions with few terms only.
template <typename St>
__device__ __forceinline__ void mma(float (&d)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                    unsigned b1) {
  if constexpr (std::is_same<St, f16_t>::value)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

}  // namespace tch
}  // namespace hdcg
