// Epilogue stores of the tensor-core GEMMs: 32 consecutive fp32 accumulator values of one output row,
// converted to the output type, optionally added to what is already there (beta = 1).
#pragma once

#include "common.cuh"
#include "tc_common.cuh"

namespace velora {

// 32 bytes in one store instruction (sm_100 has 256-bit global stores).  A thread of the epilogue owns a
// contiguous piece of ONE output row, so 16-byte stores touch every 32-byte sector twice, from two
// instructions, and L2 counts two sector writes: on a product that is all epilogue (tiny K) ncu showed
// 4.19 M sector writes for 2.10 M sectors of output and the L2 at 65 % of its throughput.
__device__ __forceinline__ void st_global_32B(void* p, const uint4& a, const uint4& b)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w) : "memory");
}

// Whether every row of an output starts on a 16-byte boundary (vector stores) or not (staged rows).
inline int c_rows_vec(const void* C, int64_t ldc, size_t elem) { return aligned16(C) && (ldc * static_cast<int64_t>(elem)) % 16 == 0; }

template <typename CT> struct Store32;
template <> struct Store32<__nv_bfloat16> {
    // 32 consecutive outputs of one row.
    static __device__ __forceinline__ void run(__nv_bfloat16* p, const uint32_t (&r)[32], int valid, int beta)
    {
        if (valid >= 32) {
            uint4* q = reinterpret_cast<uint4*>(p);
            uint4 o[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float f[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) f[e] = __uint_as_float(r[8 * i + e]);
                if (beta) {
                    const uint4 old = q[i];
                    f[0] += bf16_lo(old.x); f[1] += bf16_hi(old.x);
                    f[2] += bf16_lo(old.y); f[3] += bf16_hi(old.y);
                    f[4] += bf16_lo(old.z); f[5] += bf16_hi(old.z);
                    f[6] += bf16_lo(old.w); f[7] += bf16_hi(old.w);
                }
                o[i].x = pack_bf16x2(f[0], f[1]);
                o[i].y = pack_bf16x2(f[2], f[3]);
                o[i].z = pack_bf16x2(f[4], f[5]);
                o[i].w = pack_bf16x2(f[6], f[7]);
            }
            if ((reinterpret_cast<uintptr_t>(p) & 31u) == 0) {
                st_global_32B(q, o[0], o[1]);
                st_global_32B(q + 2, o[2], o[3]);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) q[i] = o[i];
            }
        } else {
#pragma unroll
            for (int e = 0; e < 32; ++e)
                if (e < valid) {
                    float f = __uint_as_float(r[e]);
                    if (beta) f += __bfloat162float(p[e]);
                    p[e] = __float2bfloat16_rn(f);
                }
        }
    }
};
template <> struct Store32<float> {
    static __device__ __forceinline__ void run(float* p, const uint32_t (&r)[32], int valid, int beta)
    {
        if (valid >= 32) {
            float4* q = reinterpret_cast<float4*>(p);
            float4 o[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                o[i] = make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]),
                                   __uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3]));
                if (beta) {
                    const float4 old = q[i];
                    o[i].x += old.x; o[i].y += old.y; o[i].z += old.z; o[i].w += old.w;
                }
            }
            if ((reinterpret_cast<uintptr_t>(p) & 31u) == 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    st_global_32B(q + 2 * i, *reinterpret_cast<const uint4*>(&o[2 * i]), *reinterpret_cast<const uint4*>(&o[2 * i + 1]));
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) q[i] = o[i];
            }
        } else {
#pragma unroll
            for (int e = 0; e < 32; ++e)
                if (e < valid) {
                    float f = __uint_as_float(r[e]);
                    if (beta) f += p[e];
                    p[e] = f;
                }
        }
    }
};

// Four consecutive outputs of a row at a multiple of four columns, rows on 16-byte boundaries.
template <typename CT> struct Store4;
template <> struct Store4<__nv_bfloat16> {
    static __device__ __forceinline__ void run(__nv_bfloat16* p, float (&y)[4], int beta)
    {
        uint2* q = reinterpret_cast<uint2*>(p);
        if (beta) {
            const uint2 old = *q;
            y[0] += bf16_lo(old.x); y[1] += bf16_hi(old.x); y[2] += bf16_lo(old.y); y[3] += bf16_hi(old.y);
        }
        *q = make_uint2(pack_bf16x2(y[0], y[1]), pack_bf16x2(y[2], y[3]));
    }
};
template <> struct Store4<float> {
    static __device__ __forceinline__ void run(float* p, float (&y)[4], int beta)
    {
        float4* q = reinterpret_cast<float4*>(p);
        if (beta) {
            const float4 old = *q;
            y[0] += old.x; y[1] += old.y; y[2] += old.z; y[3] += old.w;
        }
        *q = make_float4(y[0], y[1], y[2], y[3]);
    }
};

// Output rows of bf16 that start on any element (odd pitch, no padding): a lane that stores its own row would touch 32
// sectors per instruction, two bytes in each.  The warp turns its 32 x 32 block over through shared memory (32 rows of
// kStagePitch floats; the odd pitch keeps both directions free of bank conflicts) and writes one row at a time,
// consecutive lanes to consecutive columns.  All lanes call; `valid` columns are the same for all of them.
constexpr int kStagePitch = 33;
constexpr int kStageFloats = 32 * kStagePitch;

template <typename CT>
__device__ __forceinline__ void store_rows_staged(CT* block, int64_t ldc, int rows, int valid, const uint32_t (&r)[32], int beta,
                                                  float* stage, int lane)
{
#pragma unroll
    for (int e = 0; e < 32; ++e) stage[lane * kStagePitch + e] = __uint_as_float(r[e]);
    __syncwarp();
    if (lane < valid) {
        CT* p = block + lane;
#pragma unroll 8
        for (int i = 0; i < 32; ++i, p += ldc) {
            if (i >= rows) break;
            float f = stage[i * kStagePitch + lane];
            if (beta) f += Elem<CT>::load(p);
            Elem<CT>::store(p, f);
        }
    }
    __syncwarp();
}

// How outputs are written: rows on odd boundaries by store_rows_staged, others by Store32 or as tiles by store_block.
enum CRows { C_ELEMENTS = 0, C_VECTORS = 1, C_TILES = 2 };

// bf16 outputs on 16-byte boundaries leave as tiles, 32 rows x 64 columns a warp: a lane that stores its own row writes 32 sectors of
// 32 lines per instruction, and a product with little else to do waits for those (8192 x 4096 with K = 16: 19.5 us, 14.0 as
// tiles, 67 MB at 4.8 TB/s; 8192 x 1024, K = 256: 9.6 and 8.1; 4096 x 4096 products of long contractions the same).  A tile
// store clips whole 16-byte chunks: where the width is no multiple of 8 the last columns' block is left to Store32.
constexpr int kStoreBytes = 32 * 128;

// A warp's 32 x 64 outputs, r[h] the columns 32 h .. of this lane's row, through its block of shared memory (128-byte swizzle) to
// C at (row0, col0).
__device__ __forceinline__ void store_block(const CUtensorMap* tmC, uint32_t block, const uint32_t (&r)[2][32], int col0, int row0, int lane)
{
    if (lane == 0) tc::bulk_wait_read();                            // the block's last content is on its way
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int k = 8 * (c % 4) + 2 * e;
            w[e] = pack_bf16x2(__uint_as_float(r[c / 4][k]), __uint_as_float(r[c / 4][k + 1]));
        }
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                     ::"r"(block + lane * 128 + ((c ^ (lane & 7)) << 4)), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
    }
    tc::fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) tc::tma_store_2d(tmC, block, col0, row0);
}

}  // namespace velora
