// CUDA-core GEMM with arbitrary element strides and fp32 accumulation.
//   C[m, n] = beta * C[m, n] + sum_k A(m, k) * B(n, k)
// It computes the dense products of Algorithm 1 (arxiv 2405.17991) for small all-fp32 ones (gemm_f32_tc.cu has the others)
// and for bf16 operands that neither TMA nor the packed copies can serve.
//
// Bound by the fp32 pipes (74 TFLOP/s at 1965 MHz).  Three shapes of the same kernel, 256 threads each:
//   128 x 128 tile, 16-deep slices, 8 x 8 outputs a thread: 64 multiply-adds for four 16-byte shared-memory loads, and
//     as packed pairs (fma.rn.f32x2, the same roundings as two single ones) half the issue slots.
//   64 x 128 tile, 4 x 8 outputs a thread, where the large one leaves most of its last wave empty.
//   64 x 64 tile, 32-deep slices, 4 x 4 outputs a thread, for outputs of few tiles; up to eight CTAs of a cluster
//     share a tile's contraction and add their partial sums through distributed shared memory in a fixed order (a
//     171 x 288 output with K = 1280 kept 15 CTAs busy for 90 us).
// 12608 x 768 x 768 in fp32: 372 us as 64 x 128 tiles, 410 as 128 x 128, 544 with scalar loads, 4 x 4 outputs and no overlap.
// Single multiply-adds instead of pairs: 455 us as 128 x 128 tiles.
// The next slice is on its way in registers while the current one is multiplied.  An operand is read with 16-byte
// loads along whichever index is contiguous where base and pitch allow, else element by element, and stored K-major.
#include <cooperative_groups.h>

#include "common.cuh"

namespace velora {
namespace {

constexpr int SG_THREADS = 256;
constexpr int SG_MAX_SPLITS = 8;                        // the portable cluster size

// How a tile of an operand is read: along K or along its rows, four elements at a time or one.
enum LoadMode { LOAD_K4 = 0, LOAD_R4 = 1, LOAD_K1 = 2, LOAD_R1 = 3 };

// A ROWS x TK tile of which every thread holds E (four or eight) elements.
template <typename T, int ROWS, int TK>
struct Tile {
    static constexpr int E = ROWS * TK / SG_THREADS;
    static_assert(ROWS * TK == E * SG_THREADS && E % 4 == 0, "whole vectors per thread");
    static __device__ __forceinline__ void load(const T* p, int64_t s_row, int64_t s_k, int64_t row0, int64_t rows,
                                                int64_t k0, int64_t k_end, int mode, float (&r)[E])
    {
        const int t = threadIdx.x;
        if (mode <= LOAD_R4) {
#pragma unroll
            for (int i = 0; i < E / 4; ++i) {
                const int idx = t + SG_THREADS * i;
                const int row = mode == LOAD_K4 ? idx / (TK / 4) : idx % (ROWS / 4) * 4;
                const int kk = mode == LOAD_K4 ? idx % (TK / 4) * 4 : idx / (ROWS / 4);
                const T* q = p + (row0 + row) * s_row + (k0 + kk) * s_k;
                const bool row_fast = mode == LOAD_R4;
                const int64_t fast_left = row_fast ? rows - (row0 + row) : k_end - (k0 + kk);
                const bool slow_in = row_fast ? k0 + kk < k_end : row0 + row < rows;
                if (sizeof(T) == 4 && slow_in && fast_left >= 4) {
                    const float4 x = *reinterpret_cast<const float4*>(q);
                    r[4 * i] = x.x; r[4 * i + 1] = x.y; r[4 * i + 2] = x.z; r[4 * i + 3] = x.w;
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e) r[4 * i + e] = (slow_in && e < fast_left) ? Elem<T>::load(q + e) : 0.f;
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < E; ++i) {
                const int idx = t + SG_THREADS * i;
                const int row = mode == LOAD_K1 ? idx / TK : idx % ROWS;
                const int kk = mode == LOAD_K1 ? idx % TK : idx / ROWS;
                r[i] = (row0 + row < rows && k0 + kk < k_end) ? Elem<T>::load(p + (row0 + row) * s_row + (k0 + kk) * s_k) : 0.f;
            }
        }
    }
    static __device__ __forceinline__ void store(float (*s)[ROWS + 4], int mode, const float (&r)[E])
    {
        const int t = threadIdx.x;
        if (mode == LOAD_K4) {
#pragma unroll
            for (int i = 0; i < E / 4; ++i) {
                const int idx = t + SG_THREADS * i;
#pragma unroll
                for (int e = 0; e < 4; ++e) s[idx % (TK / 4) * 4 + e][idx / (TK / 4)] = r[4 * i + e];
            }
        } else if (mode == LOAD_R4) {
#pragma unroll
            for (int i = 0; i < E / 4; ++i) {
                const int idx = t + SG_THREADS * i;
                *reinterpret_cast<float4*>(&s[idx / (ROWS / 4)][idx % (ROWS / 4) * 4]) =
                    make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < E; ++i) {
                const int idx = t + SG_THREADS * i;
                if (mode == LOAD_K1) s[idx % TK][idx / TK] = r[i];
                else s[idx / ROWS][idx % ROWS] = r[i];
            }
        }
    }
};

// Two multiply-adds, each rounded as the single instruction rounds.
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ float2 unpack2(unsigned long long d)
{
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(d));
    return f;
}

template <typename CT>
__device__ __forceinline__ void put4(CT* __restrict__ C, int64_t ldc, int beta, int64_t m, int64_t n, int64_t Mdim, int64_t Ndim,
                                     const float (&x)[4], int c_vec)
{
    if (m >= Mdim || n >= Ndim) return;
    CT* p = C + m * ldc + n;
    if (sizeof(CT) == 4 && c_vec && n + 4 <= Ndim) {
        float4* q = reinterpret_cast<float4*>(p);
        float4 o = make_float4(x[0], x[1], x[2], x[3]);
        if (beta) {
            const float4 old = *q;
            o.x += old.x; o.y += old.y; o.z += old.z; o.w += old.w;
        }
        *q = o;
        return;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (n + e < Ndim) {
            float f = x[e];
            if (beta) f += Elem<CT>::load(p + e);
            Elem<CT>::store(p + e, f);
        }
}

__host__ __device__ constexpr int slice_depth(int gm, int gn) { return gm * gn == 1 ? 32 : 16; }

// GM groups of four rows and GN of four columns per thread, 64 apart: a tile of 64 * GM x 64 * GN.  gridDim.z = CTAs that
// share a tile's contraction (a cluster; 64 x 64 tiles only).
template <int GM, int GN, typename AT, typename BT, typename CT>
__global__ void __launch_bounds__(SG_THREADS, 2)
gemm_simt_kernel(const AT* A, int64_t a_sm, int64_t a_sk, int a_mode,
                 const BT* B, int64_t b_sn, int64_t b_sk, int b_mode,
                 CT* __restrict__ C, int64_t ldc, int beta, int c_vec,
                 int64_t Mdim, int64_t Ndim, int64_t Kdim, int64_t k_per_split)
{
    constexpr int TM = 64 * GM, TN = 64 * GN, TK = slice_depth(GM, GN);
    __shared__ __align__(16) float As[2][TK][TM + 4];
    __shared__ __align__(16) float Bs[2][TK][TN + 4];
    const int t = threadIdx.x;
    const int tx = t % 16, ty = t / 16;
    const int64_t m0 = static_cast<int64_t>(blockIdx.y) * TM;
    const int64_t n0 = static_cast<int64_t>(blockIdx.x) * TN;
    const int64_t k_begin = blockIdx.z * k_per_split;
    const int64_t k_end = k_begin + k_per_split < Kdim ? k_begin + k_per_split : Kdim;

    unsigned long long acc[4 * GM][2 * GN];
#pragma unroll
    for (int i = 0; i < 4 * GM; ++i)
#pragma unroll
        for (int j = 0; j < 2 * GN; ++j) acc[i][j] = 0ull;       // two zeros

    pdl_wait();
    if (gridDim.z == 1) pdl_trigger();
    float ra[Tile<AT, TM, TK>::E], rb[Tile<BT, TN, TK>::E];
    Tile<AT, TM, TK>::load(A, a_sm, a_sk, m0, Mdim, k_begin, k_end, a_mode, ra);
    Tile<BT, TN, TK>::load(B, b_sn, b_sk, n0, Ndim, k_begin, k_end, b_mode, rb);
    Tile<AT, TM, TK>::store(As[0], a_mode, ra);
    Tile<BT, TN, TK>::store(Bs[0], b_mode, rb);
    __syncthreads();
    int buf = 0;
    for (int64_t k0 = k_begin; k0 < k_end; k0 += TK, buf ^= 1) {
        const bool more = k0 + TK < k_end;
        if (more) {
            Tile<AT, TM, TK>::load(A, a_sm, a_sk, m0, Mdim, k0 + TK, k_end, a_mode, ra);
            Tile<BT, TN, TK>::load(B, b_sn, b_sk, n0, Ndim, k0 + TK, k_end, b_mode, rb);
        }
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            float a[4 * GM];
            unsigned long long b[2 * GN];
#pragma unroll
            for (int g = 0; g < GM; ++g) {
                const float4 x = *reinterpret_cast<const float4*>(&As[buf][kk][64 * g + ty * 4]);
                a[4 * g] = x.x; a[4 * g + 1] = x.y; a[4 * g + 2] = x.z; a[4 * g + 3] = x.w;
            }
#pragma unroll
            for (int g = 0; g < GN; ++g) {
                const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][64 * g + tx * 4]);
                b[2 * g] = y.x; b[2 * g + 1] = y.y;
            }
#pragma unroll
            for (int i = 0; i < 4 * GM; ++i) {
                const unsigned long long aa = pack2(a[i], a[i]);
#pragma unroll
                for (int j = 0; j < 2 * GN; ++j) fma2(acc[i][j], aa, b[j]);
            }
        }
        if (more) {
            Tile<AT, TM, TK>::store(As[buf ^ 1], a_mode, ra);
            Tile<BT, TN, TK>::store(Bs[buf ^ 1], b_mode, rb);
        }
        __syncthreads();
    }

    if constexpr (GM * GN == 1) if (gridDim.z > 1) {
        namespace cg = cooperative_groups;
        cg::cluster_group cluster = cg::this_cluster();
        float* mine = &As[0][0][0];                             // 64 rows of TM + 4 floats: the slices have been used up
        static_assert(2 * TK >= 64, "the partial tile fits in As");
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 lo = unpack2(acc[i][0]), hi = unpack2(acc[i][1]);
            *reinterpret_cast<float4*>(mine + (ty * 4 + i) * (TM + 4) + tx * 4) = make_float4(lo.x, lo.y, hi.x, hi.y);
        }
        cluster.sync();
        const int splits = static_cast<int>(gridDim.z), rows_per = 64 / splits;     // a power of two
        for (int idx = t; idx < rows_per * 16; idx += SG_THREADS) {
            const int row = static_cast<int>(blockIdx.z) * rows_per + idx / 16, col = idx % 16 * 4;
            float x[4] = {0.f, 0.f, 0.f, 0.f};
            float4 part[SG_MAX_SPLITS];
#pragma unroll
            for (int s = 0; s < SG_MAX_SPLITS; ++s)
                if (s < splits) part[s] = *reinterpret_cast<const float4*>(cluster.map_shared_rank(mine, s) + row * (TM + 4) + col);
#pragma unroll
            for (int s = 0; s < SG_MAX_SPLITS; ++s)             // fixed order
                if (s < splits) { x[0] += part[s].x; x[1] += part[s].y; x[2] += part[s].z; x[3] += part[s].w; }
            put4<CT>(C, ldc, beta, m0 + row, n0 + col, Mdim, Ndim, x, c_vec);
        }
        cluster.sync();                                          // nobody leaves while its partial is still being read
        return;
    }
#pragma unroll
    for (int i = 0; i < 4 * GM; ++i)
#pragma unroll
        for (int g = 0; g < GN; ++g) {
            const float2 lo = unpack2(acc[i][2 * g]), hi = unpack2(acc[i][2 * g + 1]);
            const float x[4] = {lo.x, lo.y, hi.x, hi.y};
            put4<CT>(C, ldc, beta, m0 + (i / 4) * 64 + ty * 4 + i % 4, n0 + 64 * g + tx * 4, Mdim, Ndim, x, c_vec);
        }
}

int load_mode(const void* p, int dtype, int64_t s_row, int64_t s_k)
{
    const bool k_fast = s_k == 1;
    const int64_t pitch = k_fast ? s_row : s_k;
    const bool vec = dtype == VELORA_F32 && aligned16(p) && pitch % 4 == 0 && (k_fast || s_row == 1);
    return k_fast ? (vec ? LOAD_K4 : LOAD_K1) : (vec ? LOAD_R4 : LOAD_R1);
}

template <int GM, int GN, typename AT, typename BT, typename CT>
int launch_tiles(const void* A, int64_t a_sm, int64_t a_sk, int a_mode, const void* B, int64_t b_sn, int64_t b_sk, int b_mode,
                 void* C, int64_t ldc, int beta, int c_vec, int64_t Mdim, int64_t Ndim, int64_t Kdim, int splits, cudaStream_t stream)
{
    constexpr int TM = 64 * GM, TN = 64 * GN, TK = slice_depth(GM, GN);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(ceil_div64(Ndim, TN)), static_cast<unsigned>(ceil_div64(Mdim, TM)), static_cast<unsigned>(splits));
    cfg.blockDim = dim3(SG_THREADS, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0] = pdl_attribute();                                  // not for clusters (common.cuh)
    if (splits > 1) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = static_cast<unsigned>(splits);
    }
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int64_t k_per_split = ceil_div64(ceil_div64(Kdim, TK), splits) * TK;
    if (cudaLaunchKernelEx(&cfg, gemm_simt_kernel<GM, GN, AT, BT, CT>, static_cast<const AT*>(A), a_sm, a_sk, a_mode,
                           static_cast<const BT*>(B), b_sn, b_sk, b_mode, static_cast<CT*>(C), ldc, beta, c_vec, Mdim, Ndim, Kdim,
                           k_per_split) != cudaSuccess) {
        cudaGetLastError();
        if (splits > 1)                                         // a refused cluster: the same tiles, one CTA each
            return launch_tiles<GM, GN, AT, BT, CT>(A, a_sm, a_sk, a_mode, B, b_sn, b_sk, b_mode, C, ldc, beta, c_vec, Mdim, Ndim, Kdim, 1, stream);
        return VELORA_ERR_CUDA;
    }
    return after_launch();
}

struct SimtShape {
    int rows, cols, splits;                                     // of a tile; CTAs that share its contraction
};

SimtShape simt_shape(int64_t Mdim, int64_t Ndim, int64_t Kdim, int sm_count)
{
    // The large tile once it gives every SM one; two of them fit on an SM.  Half of it in rows where that saves more of the
    // last wave than its extra loads cost: 12608 x 768 is 594 large tiles on 296 places, two of which ran alone for a third
    // of the time, and 1182 half tiles (layer of two such products: 887 -> 813 us).
    const int64_t large = ceil_div64(Mdim, 128) * ceil_div64(Ndim, 128), half = ceil_div64(Mdim, 64) * ceil_div64(Ndim, 128);
    if (large >= sm_count) {
        const int64_t places = 2 * static_cast<int64_t>(sm_count);
        if (11 * ceil_div64(half, places) < 20 * ceil_div64(large, places)) return SimtShape{64, 128, 1};
        return SimtShape{128, 128, 1};
    }
    // Few small tiles: share the contraction while that leaves every CTA four slices and no more than two CTAs per SM.
    const int64_t tiles = ceil_div64(Mdim, 64) * ceil_div64(Ndim, 64);
    int splits = 1;
    while (splits < SG_MAX_SPLITS && tiles * splits * 2 <= 2 * sm_count && ceil_div64(Kdim, 32) >= 8 * splits) splits *= 2;
    return SimtShape{64, 64, splits};
}

template <typename AT, typename BT, typename CT>
int dispatch_tiles(const void* A, int a_dtype, int64_t a_sm, int64_t a_sk, const void* B, int b_dtype, int64_t b_sn, int64_t b_sk,
                   void* C, int c_dtype, int64_t ldc, int beta, int64_t Mdim, int64_t Ndim, int64_t Kdim, cudaStream_t stream)
{
    DeviceInfo di;
    const int rc = device_info(&di);
    if (rc != VELORA_OK) return rc;
    const int a_mode = load_mode(A, a_dtype, a_sm, a_sk), b_mode = load_mode(B, b_dtype, b_sn, b_sk);
    const int c_vec = c_dtype == VELORA_F32 && aligned16(C) && ldc % 4 == 0;
    const SimtShape shape = simt_shape(Mdim, Ndim, Kdim, di.sm_count);
    if (shape.rows == 128)
        return launch_tiles<2, 2, AT, BT, CT>(A, a_sm, a_sk, a_mode, B, b_sn, b_sk, b_mode, C, ldc, beta, c_vec, Mdim, Ndim, Kdim, 1, stream);
    if (shape.cols == 128)
        return launch_tiles<1, 2, AT, BT, CT>(A, a_sm, a_sk, a_mode, B, b_sn, b_sk, b_mode, C, ldc, beta, c_vec, Mdim, Ndim, Kdim, 1, stream);
    return launch_tiles<1, 1, AT, BT, CT>(A, a_sm, a_sk, a_mode, B, b_sn, b_sk, b_mode, C, ldc, beta, c_vec, Mdim, Ndim, Kdim, shape.splits, stream);
}

}  // namespace

// Waves of CTAs, each its share of K at what a step of its tile takes on a full chip; a cluster costs its launch and the exchange.
double gemm_simt_f32_us(int64_t Mdim, int64_t Ndim, int64_t Kdim, int sm_count)
{
    const SimtShape t = simt_shape(Mdim, Ndim, Kdim, sm_count);
    const int64_t ctas = ceil_div64(Mdim, t.rows) * ceil_div64(Ndim, t.cols) * t.splits;
    const double step = t.rows == 128 ? 0.22 : (t.cols == 128 ? 0.121 : 0.061);
    return (t.splits > 1 ? 9.0 : 5.0) + ceil_div64(ctas, 2 * static_cast<int64_t>(sm_count)) * step * ceil_div64(Kdim, t.splits);
}

int launch_gemm_simt(const void* A, int a_dtype, int64_t a_sm, int64_t a_sk,
                     const void* B, int b_dtype, int64_t b_sn, int64_t b_sk,
                     void* C, int c_dtype, int64_t ldc, int beta,
                     int64_t Mdim, int64_t Ndim, int64_t Kdim, cudaStream_t stream)
{
    if (Mdim <= 0 || Ndim <= 0) return VELORA_OK;
    if (ceil_div64(Mdim, 64) > 65535) return VELORA_ERR_UNSUPPORTED;
#define VELORA_SIMT_CASE(AT, BT)                                                                                                  \
    return c_dtype == VELORA_BF16                                                                                                 \
               ? dispatch_tiles<AT, BT, __nv_bfloat16>(A, a_dtype, a_sm, a_sk, B, b_dtype, b_sn, b_sk, C, c_dtype, ldc, beta, Mdim, Ndim, Kdim, stream) \
               : dispatch_tiles<AT, BT, float>(A, a_dtype, a_sm, a_sk, B, b_dtype, b_sn, b_sk, C, c_dtype, ldc, beta, Mdim, Ndim, Kdim, stream)
    if (b_dtype == VELORA_FP8_E4M3) {                    // Z in its 8-bit store as the second operand of dY^T Z
        if (a_dtype == VELORA_BF16) { VELORA_SIMT_CASE(__nv_bfloat16, e4m3_t); }
        VELORA_SIMT_CASE(float, e4m3_t);
    }
    if (a_dtype == VELORA_BF16 && b_dtype == VELORA_BF16) { VELORA_SIMT_CASE(__nv_bfloat16, __nv_bfloat16); }
    if (a_dtype == VELORA_BF16 && b_dtype == VELORA_F32) { VELORA_SIMT_CASE(__nv_bfloat16, float); }
    if (a_dtype == VELORA_F32 && b_dtype == VELORA_BF16) { VELORA_SIMT_CASE(float, __nv_bfloat16); }
    VELORA_SIMT_CASE(float, float);
#undef VELORA_SIMT_CASE
}

}  // namespace velora
