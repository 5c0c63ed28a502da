// FP16 tensor-core helpers: ldmatrix, mma.sync with FP32 accumulation, and FP32 values split into
// two FP16 parts under a common power-of-two scale.
//
// The split: a group of values is scaled so that its largest lies in [2^14, 2^15); a scaled value a
// is h + 2^-12 l with h = fp16(a) and l = fp16(2^12 (a - h)).  h and l keep 11 bits each, so the pair
// keeps 22, as a TF32 high / low pair does, for every value down to 2^-29 of the group's
// largest; a smaller one keeps an absolute 2^-51 of the largest.  The low part has a scale of its
// own because at h's scale it would turn subnormal from 2^-17 on.  Products with h and with l
// accumulate apart and meet as h + 2^-12 l.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

namespace dwf {

// four 8 x 8 tiles of halves: lane l gives the address of row l % 8 of tile l / 8
template <bool TRANS>
__device__ __forceinline__ void ldmatrix4(uint32_t (&a)[4], uint32_t addr) {
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(addr) : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(addr) : "memory");
}

// c += a b, k = 16.  Fragments (lane = 4 g + t): a0 (row g, k 2 t, + 1), a1 (g + 8, 2 t), a2 (g, 2 t + 8),
// a3 (g + 8, 2 t + 8); b0 (k 2 t, + 1, column g), b1 (2 t + 8); c0 (g, 2 t), c1 (g, 2 t + 1), c2, c3 (g + 8)
__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// c = a b
__device__ __forceinline__ void mma_f16_zero(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                             uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%10,%10,%10,%10};"
                 : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
// c += a b, k = 8: the first half of the fragments above
__device__ __forceinline__ void mma_f16_k8(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(b0));
}

constexpr float F16_LOW = 1.f / 4096.f;    // the scale of a low part

// The scale of a group whose largest magnitude is m, and what undoes it.  Groups below 2^-112 are left
// where 2^126 brings them.
__device__ __forceinline__ void f16_scale(float m, float& scale, float& back) {
    const int e = max((int)(__float_as_uint(m) >> 23), 15);
    scale = __uint_as_float((unsigned)(127 + 14 + 127 - e) << 23);
    back = __uint_as_float((unsigned)(e - 14) << 23);
}
__device__ __forceinline__ void f16_split(float a, float b, __half2& h, __half2& l) {
    h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    l = __floats2half2_rn((a - f.x) * 4096.f, (b - f.y) * 4096.f);
}

}  // namespace dwf
