// An fp32 number as the sum of three bf16 numbers, x = h + m + l: exact (8 + 8 + 8 significant bits) but for numbers that round to
// infinity in bf16, infinities and NaN (no finite h or m) and numbers below 2^-110 (the last bits of l, at most 2^-134, are lost).
#pragma once

#include "common.cuh"

namespace velora {

// x less the two bf16 numbers nearest to it: exact, the remainder has 16 significant bits the first time and 8 the second.
__device__ __forceinline__ float2 minus_parts(float2 x, uint32_t parts)
{
    float2 r;
    asm("{\n\t.reg .b64 x, h, n;\n\t"
        "mov.b64 x, {%2, %3};\n\tmov.b64 h, {%4, %5};\n\tmov.b64 n, {%6, %6};\n\t"
        "fma.rn.f32x2 x, h, n, x;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(x.x), "f"(x.y), "f"(bf16_lo(parts)), "f"(bf16_hi(parts)), "f"(-1.f));
    return r;
}

// True for an output that the split may have got wrong (not finite, or so small altogether that vanished last parts could show); zero is right either way, since the products
// that vanish then are below the smallest fp32 number.
__device__ __forceinline__ bool split_suspect(float x)
{
    const float a = fabsf(x);
    return !(a <= 3.402823466e+38f) || (a < 5.421010862e-20f && a != 0.f);
}

// The same for many outputs at once, two instructions each.
struct SplitCheck {
    float finite = 0.f;                  // NaN once an output is not finite
    uint32_t least = 0xffffffffu;        // twice the bits of the smallest magnitude less one: zero, which is right, counts as the largest
    __device__ __forceinline__ void add(float x)
    {
        finite = fmaf(x, 0.f, finite);
        least = min(least, 2u * __float_as_uint(x) - 1u);
    }
    __device__ __forceinline__ bool suspect() const { return finite != 0.f || least < 2u * 0x1f800000u - 1u; }      // 2^-64
};

}  // namespace velora
