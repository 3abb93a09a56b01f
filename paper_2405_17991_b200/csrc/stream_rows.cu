// Row-streaming kernels for sub-tokens of Dsub = 8 * 2^k (8 .. 1024) elements: compress (arxiv 2405.17991, Section 3.1
// Eq. 1) and the partial sums of init_v (Section 3.2).  A lane takes chunks of VEC consecutive elements, 16 bytes of bf16
// (VEC = 8) or fp32 (VEC = 4) where the rows are 16-byte aligned, single elements where they are not: a warp's load then
// still covers 32 consecutive elements, and nothing but the width of the load changes.  Against one warp per sub-token
// with one load in flight, compress took 6.5 us instead of 47 on 12608 x 768 fp32 (Dsub 32) and 74 instead of 244 on 8192 x
// 11005 unpadded bf16 (Dsub 64), the sub-token sum 77 instead of 308 there.
//
// Both are bound by the one pass over X, so the kernel is as plain as a read stream can be: a warp owns a
// token row and walks it in rounds of U = 8 load instructions, each of which reads one contiguous 512-byte
// span (32 lanes x 16 bytes = 32 chunks of 8 elements); all eight are issued before the first is used.  With
// 8 CTAs of 256 threads per SM that keeps 128-256 KB per SM in flight with no shared memory, no barrier and
// no set-up to speak of -- measured against a TMA-fed shared-memory ring (three 32 KB stages per CTA, two
// CTAs per SM) this form is faster by about 4 us per call on a 67 MB input and by 2 us on a 180 MB one, and
// runs within a few per cent of a kernel that only reads.
//
// A sub-token of length Dsub = VEC * L covers L consecutive chunks: LPS = min(L, 32) adjacent lanes hold one
// part of it, and for L > 32 the CH = L / 32 consecutive load instructions of a round complete it.  A lane's
// position inside the sub-token never changes (rounds advance by multiples of 32 * CH chunks), so its slice
// of v lives in registers.  compress: fp32 products and sums, xor-shuffle reduction over the LPS lanes,
// the lane at position 0 stores Z[row, m].  init_v: the lane adds what it loads into VEC * CH running sums; the
// CTA then adds the sums of the lanes that share a position in a fixed order and writes one row of partials.
//
// Fewer rows than warps: a row is cut into runs of whole rounds, one warp each.  16 rows of 11005 unpadded bf16 elements with Dsub 64:
// compress 2 us, 17 with a warp per row; the sub-token sum 7 us, 14.
//
// Columns at or beyond D count as zeros: chunks past the row's end are not loaded and a last chunk that
// straddles D is masked, which is the zero extension of a ragged last sub-token.
#include "common.cuh"
#include "gemm_tc.cuh"

namespace velora {
namespace {

constexpr int RW_THREADS = 256;
constexpr int RW_WARPS = RW_THREADS / 32;
constexpr int RW_U = 8;                          // load instructions in flight per warp

template <typename ZT> __device__ __forceinline__ void put_z(ZT* p, float z);
template <> __device__ __forceinline__ void put_z<float>(float* p, float z) { *p = z; }
template <> __device__ __forceinline__ void put_z<__nv_bfloat16>(__nv_bfloat16* p, float z) { *p = __float2bfloat16_rn(z); }
template <> __device__ __forceinline__ void put_z<e4m3_t>(e4m3_t* p, float z) { *p = float_to_e4m3(z); }

// Chunk c of a row as loaded (KEEP: a compress of the same rows is likely to follow, so they
// are left in L2), and its VEC values; zeros beyond column D.  full = D / VEC whole chunks, tail = D % VEC.
template <typename XT, int VEC> struct Chunk;
template <> struct Chunk<__nv_bfloat16, 8> {
    typedef uint4 Raw;
    template <bool KEEP>
    static __device__ __forceinline__ Raw load(const __nv_bfloat16* row, int c, int full, int tail)
    {
        const uint4* q = reinterpret_cast<const uint4*>(row) + c;
        // A last partial chunk lies inside the row's pitch (a multiple of 8 elements).
        const bool take = c < full || (c == full && tail);
        uint4 x = make_uint4(0u, 0u, 0u, 0u);
        if (!KEEP) x = ld_stream_if(q, take);
        else if (take) x = *q;
        if (c == full && tail) {
            uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (2 * i >= tail) w[i] = 0u;
                else if (2 * i + 1 >= tail) w[i] &= 0x0000ffffu;
            }
            x = make_uint4(w[0], w[1], w[2], w[3]);
        }
        return x;
    }
    static __device__ __forceinline__ void unpack(const Raw& d, float (&x)[8])
    {
        x[0] = bf16_lo(d.x); x[1] = bf16_hi(d.x);
        x[2] = bf16_lo(d.y); x[3] = bf16_hi(d.y);
        x[4] = bf16_lo(d.z); x[5] = bf16_hi(d.z);
        x[6] = bf16_lo(d.w); x[7] = bf16_hi(d.w);
    }
};
template <> struct Chunk<float, 4> {
    typedef float4 Raw;
    template <bool KEEP>
    static __device__ __forceinline__ Raw load(const float* row, int c, int full, int tail)
    {
        const float4* q = reinterpret_cast<const float4*>(row) + c;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (KEEP) {
            if (c < full) x = *q;
        } else {
            const uint4 w = ld_stream_if(q, c < full);
            x = make_float4(__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w));
        }
        if (c == full && tail) {                 // the row may end inside the chunk and so may the buffer
            x.x = row[4 * c];
            if (tail > 1) x.y = row[4 * c + 1];
            if (tail > 2) x.z = row[4 * c + 2];
        }
        return x;
    }
    static __device__ __forceinline__ void unpack(const Raw& d, float (&x)[4]) { x[0] = d.x; x[1] = d.y; x[2] = d.z; x[3] = d.w; }
};
template <typename XT> struct Chunk<XT, 1> {
    typedef XT Raw;
    template <bool KEEP>
    static __device__ __forceinline__ Raw load(const XT* row, int c, int full, int)
    {
        return c < full ? row[c] : static_cast<XT>(0.f);
    }
    static __device__ __forceinline__ void unpack(const Raw& d, float (&x)[1]) { x[0] = static_cast<float>(d); }
};

template <typename XT, int VEC, int LPS, int CH, bool INIT, typename ZT>
__global__ void __launch_bounds__(RW_THREADS)
stream_rows_kernel(const XT* X, int N, int D, int64_t ldx, int M, int segs, int seg_rounds,
                   const float* v, ZT* __restrict__ Z, int64_t ldz, float* __restrict__ partials)
{
    constexpr int U = CH > RW_U ? CH : RW_U;
    static_assert(CH == 1 || LPS == 32, "several chunks per lane only for sub-tokens wider than a warp's span");
    static_assert(U % CH == 0, "a round must hold whole sub-tokens");
    typedef Chunk<XT, VEC> C;
    // Programmatic stream serialisation (common.cuh): resident early, nothing read or written before the wait.
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int q = lane & (LPS - 1);               // position of this lane's chunk inside a 32-chunk part
    const int full = D / VEC, tail = D % VEC;
    const int cpr = full + (tail ? 1 : 0);        // chunks that hold data

    float vr[CH][VEC];                            // compress: slice of v; init_v: running sums
#pragma unroll
    for (int i = 0; i < CH; ++i)
#pragma unroll
        for (int e = 0; e < VEC; ++e) vr[i][e] = INIT ? 0.f : v[VEC * (q + LPS * i) + e];

    // compress goes through the rows from the last to the first: whatever read or wrote X before it went the other way, so the
    // last rows are the ones still in L2 (a 180 MB X right behind its sub-token sum: 32 -> 23 us).
    const int warps = gridDim.x * RW_WARPS;
    const int items = N * segs;                   // runs of seg_rounds rounds (segs == 1: whole rows)
    for (int at = blockIdx.x * RW_WARPS + (threadIdx.x >> 5); at < items; at += warps) {
        const int item = INIT ? at : items - 1 - at;
        const int row = segs == 1 ? item : item / segs;
        const XT* rp = X + static_cast<int64_t>(row) * ldx;
        ZT* zrow = INIT ? nullptr : Z + static_cast<int64_t>(row) * ldz;
        int left = full, end = cpr, M_left = M;   // whole chunks, chunks to walk and sub-tokens from where the run starts
        if (segs > 1) {
            const int c_begin = (item - row * segs) * seg_rounds * (32 * U), m_begin = c_begin / (LPS * CH);
            rp += c_begin * VEC;
            if (!INIT) zrow += m_begin;
            left -= c_begin;
            M_left -= m_begin;
            end = cpr - c_begin < seg_rounds * (32 * U) ? cpr - c_begin : seg_rounds * (32 * U);
        }
        for (int c0 = 0; c0 < end; c0 += 32 * U) {
            typename C::Raw d[U];
#pragma unroll
            for (int u = 0; u < U; ++u) d[u] = C::template load<INIT>(rp, c0 + 32 * u + lane, left, tail);
            float part = 0.f;                     // CH > 1: sum over the parts of one sub-token so far
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = u % CH;             // which part of the sub-token this instruction read
                float x[VEC];
                C::unpack(d[u], x);
                if (INIT) {
#pragma unroll
                    for (int e = 0; e < VEC; ++e) vr[i][e] += x[e];
                } else {
                    float a0 = x[0] * vr[i][0], a1 = 0.f;
                    if (VEC > 1) a1 = x[1 % VEC] * vr[i][1 % VEC];
#pragma unroll
                    for (int e = 2; e < VEC; e += 2) {
                        a0 = fmaf(x[e], vr[i][e], a0);
                        a1 = fmaf(x[e + 1], vr[i][e + 1], a1);
                    }
                    part = (i == 0) ? a0 + a1 : part + (a0 + a1);
                    if (i == CH - 1) {
                        float k = part;
#pragma unroll
                        for (int off = LPS / 2; off >= 1; off >>= 1) k += __shfl_xor_sync(0xffffffffu, k, off);
                        // first chunk of the sub-token: c0 + 32 * (u - i); its index m = that / (LPS * CH) (+ lane / LPS)
                        const int m = (c0 + 32 * (u - i)) / (LPS * CH) + (CH == 1 ? lane / LPS : 0);
                        if (q == 0 && m < M_left) put_z<ZT>(zrow + m, k);
                    }
                }
            }
        }
    }

    if constexpr (INIT) {
        // Fixed-order sum over the lanes of the CTA that share a position.
        __shared__ float sacc[RW_THREADS * VEC * CH];
#pragma unroll
        for (int i = 0; i < CH; ++i)
#pragma unroll
            for (int e = 0; e < VEC; ++e) sacc[(threadIdx.x * CH + i) * VEC + e] = vr[i][e];
        __syncthreads();
        constexpr int Dsub = VEC * LPS * CH;
        for (int j = threadIdx.x; j < Dsub; j += RW_THREADS) {
            const int chunk = j / VEC, e = j % VEC;
            const int qq = chunk % LPS, i = chunk / LPS;
            float sum = 0.f;
            for (int t = qq; t < RW_THREADS; t += LPS) sum += sacc[(t * CH + i) * VEC + e];
            partials[static_cast<int64_t>(blockIdx.x) * Dsub + j] = sum;
        }
    }
}

struct RowsPlan {
    bool ok;
    int vec, lps, ch, M, segs, seg_rounds, grid;
};

RowsPlan plan_rows(const void* X, int x_dtype, int64_t N, int64_t D, int64_t ldx, int Dsub, int sm_count, int max_grid, bool sum)
{
    RowsPlan p{};
    if (Dsub < 8 || Dsub > 1024 || (Dsub & (Dsub - 1))) return p;
    if (N < 1 || N >= (1 << 30) || D >= (1 << 30)) return p;
    const int wide = x_dtype == VELORA_BF16 ? 8 : 4;
    p.vec = aligned16(X) && ldx % wide == 0 ? wide : 1;
    const int L = Dsub / p.vec;
    p.lps = L < 32 ? L : 32;
    p.ch = L / p.lps;
    p.M = static_cast<int>(ceil_div64(D, Dsub));
    int64_t cap = static_cast<int64_t>(sm_count) * kStreamCtasPerSm;
    if (max_grid > 0 && cap > max_grid) cap = max_grid;
    // Rows are cut while there are two warps and more for each; for the sub-token sum of four warps per SM, because each CTA adds
    // a row to what the finalize kernel's one CTA adds up (512 x 2045 fp32, Dsub 256: 16 us with as many runs as compress).
    const int64_t rounds = ceil_div64(ceil_div64(D, p.vec), 32 * (p.ch > RW_U ? p.ch : RW_U));
    const int64_t wanted = sum ? 4 * static_cast<int64_t>(sm_count) : cap * RW_WARPS;
    int64_t segs = N < wanted ? wanted / N : 1;
    if (segs > rounds) segs = rounds;
    p.seg_rounds = static_cast<int>(ceil_div64(rounds, segs));
    p.segs = static_cast<int>(ceil_div64(rounds, p.seg_rounds));
    const int64_t grid = ceil_div64(N * p.segs, RW_WARPS);
    p.grid = static_cast<int>(grid < cap ? grid : cap);
    p.ok = true;
    return p;
}

template <typename XT, int VEC, int LPS, int CH, bool INIT, typename ZT>
int launch_rows(const RowsPlan& p, const void* X, int64_t N, int64_t D, int64_t ldx, const float* v, ZT* Z, int64_t ldz,
                float* partials, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(p.grid), 1, 1);
    cfg.blockDim = dim3(RW_THREADS, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr = pdl_attribute();
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, stream_rows_kernel<XT, VEC, LPS, CH, INIT, ZT>, static_cast<const XT*>(X), static_cast<int>(N),
                           static_cast<int>(D), ldx, p.M, p.segs, p.seg_rounds, v, Z, ldz, partials) != cudaSuccess) {
        cudaGetLastError();
        return VELORA_ERR_CUDA;
    }
    return after_launch();
}

template <bool INIT, typename ZT>
int dispatch_rows(const RowsPlan& p, const void* X, int x_dtype, int64_t N, int64_t D, int64_t ldx, const float* v, ZT* Z, int64_t ldz,
                  float* partials, cudaStream_t stream)
{
#define VELORA_ROWS_CASE(XT, VECV, LPSV, CHV) \
    if (p.vec == VECV && p.lps == LPSV && p.ch == CHV) \
        return launch_rows<XT, VECV, LPSV, CHV, INIT, ZT>(p, X, N, D, ldx, v, Z, ldz, partials, stream)
#define VELORA_ROWS_ONE(XT) \
    VELORA_ROWS_CASE(XT, 1, 8, 1); VELORA_ROWS_CASE(XT, 1, 16, 1); VELORA_ROWS_CASE(XT, 1, 32, 1); VELORA_ROWS_CASE(XT, 1, 32, 2); \
    VELORA_ROWS_CASE(XT, 1, 32, 4); VELORA_ROWS_CASE(XT, 1, 32, 8); VELORA_ROWS_CASE(XT, 1, 32, 16); VELORA_ROWS_CASE(XT, 1, 32, 32)
    if (x_dtype == VELORA_BF16) {
        VELORA_ROWS_CASE(__nv_bfloat16, 8, 1, 1);
        VELORA_ROWS_CASE(__nv_bfloat16, 8, 2, 1);
        VELORA_ROWS_CASE(__nv_bfloat16, 8, 4, 1);
        VELORA_ROWS_CASE(__nv_bfloat16, 8, 8, 1);
        VELORA_ROWS_CASE(__nv_bfloat16, 8, 16, 1);
        VELORA_ROWS_CASE(__nv_bfloat16, 8, 32, 1);
        VELORA_ROWS_CASE(__nv_bfloat16, 8, 32, 2);
        VELORA_ROWS_CASE(__nv_bfloat16, 8, 32, 4);
        VELORA_ROWS_ONE(__nv_bfloat16);
    } else {
        VELORA_ROWS_CASE(float, 4, 2, 1);
        VELORA_ROWS_CASE(float, 4, 4, 1);
        VELORA_ROWS_CASE(float, 4, 8, 1);
        VELORA_ROWS_CASE(float, 4, 16, 1);
        VELORA_ROWS_CASE(float, 4, 32, 1);
        VELORA_ROWS_CASE(float, 4, 32, 2);
        VELORA_ROWS_CASE(float, 4, 32, 4);
        VELORA_ROWS_CASE(float, 4, 32, 8);
        VELORA_ROWS_ONE(float);
    }
#undef VELORA_ROWS_ONE
#undef VELORA_ROWS_CASE
    return VELORA_ERR_UNSUPPORTED;
}

}  // namespace

int launch_compress_rows(const void* X, int x_dtype, int64_t N, int64_t D, int64_t ldx, int Dsub, const float* v,
                         void* Z, int z_dtype, int64_t ldz, cudaStream_t stream)
{
    DeviceInfo di;
    const int rc = device_info(&di);
    if (rc != VELORA_OK) return rc;
    const RowsPlan p = plan_rows(X, x_dtype, N, D, ldx, Dsub, di.sm_count, 0, false);
    if (!p.ok) return VELORA_ERR_UNSUPPORTED;
    if (z_dtype == VELORA_F32)
        return dispatch_rows<false, float>(p, X, x_dtype, N, D, ldx, v, static_cast<float*>(Z), ldz, nullptr, stream);
    if (z_dtype == VELORA_FP8_E4M3)
        return dispatch_rows<false, e4m3_t>(p, X, x_dtype, N, D, ldx, v, static_cast<e4m3_t*>(Z), ldz, nullptr, stream);
    return dispatch_rows<false, __nv_bfloat16>(p, X, x_dtype, N, D, ldx, v, static_cast<__nv_bfloat16*>(Z), ldz, nullptr, stream);
}

int launch_init_v_partials_rows(const void* X, int x_dtype, int64_t N, int64_t D, int64_t ldx, int Dsub,
                                float* partials, int max_partials, int* num_partials, cudaStream_t stream)
{
    DeviceInfo di;
    const int rc = device_info(&di);
    if (rc != VELORA_OK) return rc;
    // Four CTAs of this kernel are resident per SM (its registers), so a grid of four per SM is one wave of CTAs
    // that each walk a few rows; a larger grid would only add partial rows for the finalize kernel to add up.
    int cap = di.sm_count * 4;
    if (max_partials > 0 && cap > max_partials) cap = max_partials;
    const RowsPlan p = plan_rows(X, x_dtype, N, D, ldx, Dsub, di.sm_count, cap, true);
    if (!p.ok) return VELORA_ERR_UNSUPPORTED;
    *num_partials = p.grid;
    return dispatch_rows<true, float>(p, X, x_dtype, N, D, ldx, nullptr, static_cast<float*>(nullptr), 0, partials, stream);
}

}  // namespace velora
