// Warp-level building blocks of the small-batch kernel: shared-memory reads, the int4 -> bf16
// expansion and the two tensor-core instructions (sparse and dense).
#pragma once
#include "common.cuh"

namespace slim {
namespace dt {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory reads by 32-bit shared address.  Plain loads, so that the compiler may move them
// ahead of the arithmetic of the previous block; the barrier waits and arrivals around a slot carry
// memory clobbers, which keeps the reads inside the slot's lifetime.
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    return *reinterpret_cast<const uint4*>(__cvta_shared_to_generic(addr));
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    return *reinterpret_cast<const uint32_t*>(__cvta_shared_to_generic(addr));
}

// D(16x8, fp32) += A(16x32 bf16, 2:4 sparse, stored 16x16) * B(32x8 bf16).
// SEL picks which thread pair of every quad supplies the metadata word.
template <int SEL>
__device__ __forceinline__ void mma_sp_16832(float* c, const uint32_t* a, const uint4& b, uint32_t e) {
    asm(
        "mma.sp::ordered_metadata.sync.aligned.m16n8k32.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9,%10,%11}, {%0,%1,%2,%3}, %12, %13;"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w), "r"(e), "n"(SEL));
}
// D(16x8, fp32) += A(16x16 bf16) * B(16x8 bf16)
__device__ __forceinline__ void mma_16816(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Two int4 codes, the first in bits 0-3 and the second in bits 16-19 of `x` (other bits
// arbitrary), as an exact bf16x2: nibble ^ 8 in the mantissa of 128.0 is 128 + (v + 8);
// subtracting 136 leaves v in [-8, 7].
__device__ __forceinline__ uint32_t nibbles_to_bf16x2(uint32_t x) {
    uint32_t y;
    asm("lop3.b32 %0, %1, %2, %3, 0x6a;" : "=r"(y) : "r"(x), "r"(0x000F000Fu), "r"(0x43084308u));
    __nv_bfloat162 v = *reinterpret_cast<__nv_bfloat162*>(&y);
    const uint32_t bias_bits = 0x43084308u;   // 136.0 twice
    v = __hsub2(v, *reinterpret_cast<const __nv_bfloat162*>(&bias_bits));
    return *reinterpret_cast<uint32_t*>(&v);
}

}  // namespace dt
}  // namespace slim
