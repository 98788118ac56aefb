// Device pieces that the selection kernels share.
#pragma once

#include "prcr_device.cuh"

namespace prcr {

// Rotation of an integer position offset: the turn fraction c * rate mod 1
// in 0.32 fixed point is bits 32..63 of the 64-bit product c * rate (rate in
// 0.64 fixed point; the product's wrap mod 2^64 keeps those bits exact for
// any int64 c), then one sin/cos evaluation on [-pi, pi).
__device__ __forceinline__ void sincos_coord(int64_t c, uint64_t turn_freq, float* s, float* co) {
    const uint64_t prod = static_cast<uint64_t>(c) * turn_freq;
    const int frac = static_cast<int>(static_cast<uint32_t>(prod >> 32));
    __sincosf(float(frac) * 1.4629180792671596e-9f, s, co);  // 2 pi / 2^32
}

// D += A B on tensor cores: mma.sync m16n8k8 with tf32 operands (the upper
// 19 bits of each float32 register), float32 accumulate. Fragments as the
// PTX ISA lays them out for this shape: a0 (row g, col t), a1 (row g + 8,
// col t), a2 (row g, col t + 4), a3 (row g + 8, col t + 4); b0 (row t, col
// g), b1 (row t + 4, col g); lane = 4 g + t.
__device__ __forceinline__ void mma_1688_tf32(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                              uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t word_of(const uint4& v, int i) {
    return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w));
}

// exp of a softmax term (x <= 0). FINE where the logits come from float32 FMAs, head
// dims other than 64 and 128 beyond small calls: __expf's error of a few units, all to
// one side, shows there. Relevances against 64 bits, __expf | expf | expf in the
// denominators alone: 16 sequences of 8192 tokens x 32 heads of 256 1.35e-7 | 1.07e-7
// | 1.19e-7, 2 of 4099 x 14 heads of 96 1.34e-7 | 1.1e-7 | 1.2e-7.
template <bool FINE>
__device__ __forceinline__ float exp_term(float x) {
    return FINE ? expf(x) : __expf(x);
}

}  // namespace prcr
