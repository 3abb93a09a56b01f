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

// What a product of split operands has to be checked for.
//   Operands: a number other than zero below 2^-110 loses up to 2^-134 ("tiny").  Where no operand is 2^30 or more ("big") that is at most
//   2^-104 a product: outputs of K * 2^-79 and more have lost 2^-25 of themselves at most.
//   Outputs: one that is not finite (operands that round to infinity in bf16, infinities, NaN), or is below 2^-120 without being zero
//   (products of last parts fall below the smallest number).
constexpr uint32_t SPLIT_TINY = 1u, SPLIT_BIG = 2u;

// Half an instruction an operand each.
struct SplitOperandCheck {
    uint32_t rests = 0;                  // what is left for the last part has its low 16 bits clear where a bf16 number holds it
    float most = 0.f;                    // NaN does not show here, but in the outputs
    __device__ __forceinline__ void add_rest(float2 x) { rests |= __float_as_uint(x.x) | __float_as_uint(x.y); }
    __device__ __forceinline__ void add(float2 x) { asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(most) : "f"(x.x), "f"(x.y)); }
    __device__ __forceinline__ uint32_t flags() const { return (rests & 0xffffu ? SPLIT_TINY : 0u) | (most >= 1073741824.f ? SPLIT_BIG : 0u); }
};

struct SplitOutputCheck {
    float finite = 0.f;                  // NaN once an output is not finite
    uint32_t least = 0xffffffffu;        // twice the bits of the smallest magnitude less one: zero counts as the largest
    float least_or_zero = 3.402823466e+38f;
    __device__ __forceinline__ void add(float x)
    {
        finite = fmaf(x, 0.f, finite);
        least = min(least, 2u * __float_as_uint(x) - 1u);
        least_or_zero = fminf(least_or_zero, fabsf(x));
    }
    __device__ __forceinline__ bool suspect(uint32_t operands, int Kdim) const
    {
        if (finite != 0.f || least < 2u * 0x03800000u - 1u) return true;
        return (operands & SPLIT_TINY) && ((operands & SPLIT_BIG) || least_or_zero < Kdim * 1.6543612251060553e-24f);       // K * 2^-79
    }
};

}  // namespace velora
