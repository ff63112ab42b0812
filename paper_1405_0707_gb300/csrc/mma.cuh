// mma.cuh -- the legacy-shape tensor-core instruction (mma.sync m16n8k16) and the bf16 splits the
// register-streamed passes use.
#pragma once
#include <stdint.h>

namespace expm {

__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// (x, y) -> three packed bf16 pairs (x in the low half): x = x0 + x1 + x2 to 2^-25 |x|
__device__ __forceinline__ void split3(float x, float y, uint32_t* u) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(u[k]) : "f"(y), "f"(x));
        if (k < 2) {
            x -= __uint_as_float(u[k] << 16);
            y -= __uint_as_float(u[k] & 0xFFFF0000u);
        }
    }
}

// The six products of two three-part operands that pass 2^-25, in the order (a part, b part): the first
// goes to the main accumulator, the others to the correction.  Callers loop over the products outermost:
// consecutive MMAs into one accumulator wait for each other (~20 clocks).
__device__ constexpr int kProdA[6] = {0, 2, 0, 1, 1, 0}, kProdB[6] = {0, 0, 2, 1, 0, 1};

}  // namespace expm
