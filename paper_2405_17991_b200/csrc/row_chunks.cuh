// Sixteen bytes at a time from rows of 16-bit elements that start anywhere.
#pragma once

#include "common.cuh"

namespace velora {

// The aligned 16 bytes at `a`; bytes outside the matrix are not touched and read as zero.
__device__ __forceinline__ uint4 load_aligned_chunk(const char* a, const char* lo_limit, const char* hi_limit)
{
    if (a >= lo_limit && a + 16 <= hi_limit) return ld_stream_if(a, true);
    uint32_t o[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int e = 0; e < 8; ++e)
        if (a + 2 * e >= lo_limit && a + 2 * e < hi_limit)
            o[e >> 1] |= static_cast<uint32_t>(*reinterpret_cast<const unsigned short*>(a + 2 * e)) << (16 * (e & 1));
    return make_uint4(o[0], o[1], o[2], o[3]);
}

// Sixteen bytes from byte s (even) of the 32 in x, y.
__device__ __forceinline__ uint4 shift_chunks(const uint4& x, const uint4& y, uint32_t s)
{
    uint32_t w[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
    if (s & 8u) {
#pragma unroll
        for (int i = 0; i < 6; ++i) w[i] = w[i + 2];
    }
    if (s & 4u) {
#pragma unroll
        for (int i = 0; i < 5; ++i) w[i] = w[i + 1];
    }
    const uint32_t bits = (s & 2u) * 8u;
    return make_uint4(__funnelshift_r(w[0], w[1], bits), __funnelshift_r(w[1], w[2], bits),
                      __funnelshift_r(w[2], w[3], bits), __funnelshift_r(w[3], w[4], bits));
}

}  // namespace velora
