// "Row of scalars times v": the write-bound half of the VeLoRA path (arxiv 2405.17991).
//   out[r, m*Dsub + j] = beta * out[r, m*Dsub + j] + (sum_s S[s][r][m]) * v[j]
// With one split and beta = 0 this is reconstruct + ungroup (Section 3.1, Eq. 2: Xhat = Z (x) v);
// with several splits it is the expansion of the factored weight gradient (dW = P (x) v, the per
// sub-token form of Section 3.2's g v v^T), where S holds partial products dY^T Z over disjoint token
// ranges that are summed here in a fixed order.
//
// A warp takes one output row and 32 consecutive sub-tokens.  Lane l loads the scalars of sub-token
// m0 + l (one coalesced load per split, all independent), then the warp walks the 32 sub-tokens,
// 32 / LPS of them per store instruction (LPS = Dsub / 8 lanes cover one sub-token), each scalar
// handed to its lanes by shuffle.  A lane keeps its 8-element slice of v in registers and its output
// pointer advances by a constant, so one store instruction costs one shuffle, eight multiplies, four
// packs and the store; every store instruction writes one contiguous 512-byte span.
//
// Fewer rows than warps: a row is cut into spans of sub-tokens, one warp each.  16 rows of 11005 unpadded bf16 elements, Dsub 64,
// added to what is there: 3 us, 111 with a warp per row.
//
// Output rows that are not 16-byte aligned take the same walk with single elements in the place of the groups of eight
// (VEC = 1): a store instruction then writes 32 consecutive elements.  8192 x 11005 unpadded bf16: 62 us, 322 with an
// integer division per element.
#include "common.cuh"

namespace velora {
namespace {

constexpr unsigned kFull = 0xffffffffu;

template <typename T> __device__ __forceinline__ float load_scalar(const T* p);
template <> __device__ __forceinline__ float load_scalar<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float load_scalar<__nv_bfloat16>(const __nv_bfloat16* p)
{
    return __bfloat162float(*p);
}
template <> __device__ __forceinline__ float load_scalar<e4m3_t>(const e4m3_t* p) { return e4m3_to_float(*p); }

template <typename WT> struct Out8;
template <> struct Out8<__nv_bfloat16> {
    static __device__ __forceinline__ void store(__nv_bfloat16* p, float (&y)[8], int beta)
    {
        uint4* q = reinterpret_cast<uint4*>(p);
        if (beta) {
            const uint4 old = *q;
            y[0] += bf16_lo(old.x); y[1] += bf16_hi(old.x);
            y[2] += bf16_lo(old.y); y[3] += bf16_hi(old.y);
            y[4] += bf16_lo(old.z); y[5] += bf16_hi(old.z);
            y[6] += bf16_lo(old.w); y[7] += bf16_hi(old.w);
        }
        uint4 o;
        o.x = pack_bf16x2(y[0], y[1]);
        o.y = pack_bf16x2(y[2], y[3]);
        o.z = pack_bf16x2(y[4], y[5]);
        o.w = pack_bf16x2(y[6], y[7]);
        __stcs(q, o);
    }
};
template <> struct Out8<float> {
    static __device__ __forceinline__ void store(float* p, float (&y)[8], int beta)
    {
        float4* q = reinterpret_cast<float4*>(p);
        if (beta) {
            const float4 a = q[0], b = q[1];
            y[0] += a.x; y[1] += a.y; y[2] += a.z; y[3] += a.w;
            y[4] += b.x; y[5] += b.y; y[6] += b.z; y[7] += b.w;
        }
        store_f32x8(p, y);
    }
};

// MODE 0: M is a multiple of 32 and Dsub divides D (no checks in the store loop).
// MODE 1: Dsub divides D, the last block of 32 sub-tokens is partial (one compare per store).
// MODE 2: ragged last sub-token as well (column checks, element-wise tail).
template <int VEC, int LPS, int CH, int MODE, typename ST, typename WT>
__global__ void __launch_bounds__(kStreamThreads)
expand_rows_vec_kernel(const ST* S, int splits, int64_t split_stride, int lds,
                       const float* v, int R, int D, int M, int segs, int span,
                       WT* __restrict__ out, int64_t ldo, int beta)
{
    static_assert(VEC == 8 || MODE == 2, "single elements are checked one by one");
    constexpr int L = LPS * CH;                  // groups of VEC elements per sub-token
    constexpr int SPW = 32 / LPS;                // sub-tokens per store instruction
    const int lane = threadIdx.x & 31;
    const int q = lane & (LPS - 1);
    const int sub = lane / LPS;
    // Programmatic stream serialisation (see common.cuh): resident early, nothing read or written before the wait.
    pdl_wait();
    pdl_trigger();
    float vr[CH][VEC];
#pragma unroll
    for (int i = 0; i < CH; ++i)
#pragma unroll
        for (int e = 0; e < VEC; ++e) vr[i][e] = v[VEC * (q + LPS * i) + e];

    // One warp per output row (or span of it) at a time.  The row's scalars are fetched for up to PB blocks of 32 sub-tokens
    // before the first store, so a row costs one load latency per PB blocks instead of one per block (a row of
    // 172 sub-tokens went through six dependent round trips to memory before).
    constexpr int PB = 4;
    const int warps = gridDim.x * (kStreamThreads / 32);
    const int items = R * segs;                  // spans of `span` sub-tokens, a multiple of SPW (segs == 1: whole rows)
    for (int item = blockIdx.x * (kStreamThreads / 32) + (threadIdx.x >> 5); item < items; item += warps) {
    const int r = segs == 1 ? item : item / segs;
    const ST* row_s = S + static_cast<int64_t>(r) * lds;
    WT* row_out = out + static_cast<int64_t>(r) * ldo;
    int end = M, M_left = M, D_left = D;         // sub-tokens to do, sub-tokens and columns from where the span starts
    if (segs > 1) {
        const int m_begin = (item - r * segs) * span;
        row_s += m_begin;
        row_out += m_begin * (L * VEC);
        M_left -= m_begin;
        D_left -= m_begin * (L * VEC);
        end = M_left < span ? M_left : span;
    }
    for (int mb0 = 0; mb0 < end; mb0 += 32 * PB) {
        float pb[PB];
#pragma unroll
        for (int b = 0; b < PB; ++b) {
            const int m = mb0 + b * 32 + lane;
            float p = 0.f;
            if (m < end) {
                const ST* sp = row_s + m;
#pragma unroll 8
                for (int s = 0; s < splits; ++s) p += load_scalar<ST>(sp + s * split_stride);   // fixed order
            }
            pb[b] = p;
        }
#pragma unroll
        for (int b = 0; b < PB; ++b) {
            const int m0 = mb0 + b * 32;
            if (m0 >= end) break;
            const int steps = (end - m0 + SPW - 1) / SPW < LPS ? (end - m0 + SPW - 1) / SPW : LPS;
            const float p = pb[b];
            // Element pointer of this lane's first chunk; each step moves on by SPW sub-tokens.
            WT* ptr = row_out + (static_cast<int64_t>(m0 + sub) * L + q) * VEC;
            if (VEC == 1 && beta && segs > 1) {
                // Few rows: eight elements of a lane at a time, what is there read first.  (With a warp per row this form takes
                // 382 us on 8192 x 11005 fp32 with Dsub 16, the one below 210.)
                constexpr int G = CH < 8 ? 8 / CH : 1;
                for (int it = 0; it < steps; it += G, ptr += G * SPW * L) {
                    float y[G][CH];
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        const int ms = (it + g) * SPW + sub;
                        const float pm = __shfl_sync(kFull, p, ms & 31);
#pragma unroll
                        for (int i = 0; i < CH; ++i) {
                            y[g][i] = pm * vr[i][0];
                            if (it + g < steps && (m0 + ms) * L + q + LPS * i < D_left) y[g][i] += Elem<WT>::load(ptr + g * SPW * L + i * LPS);
                        }
                    }
#pragma unroll
                    for (int g = 0; g < G; ++g)
#pragma unroll
                        for (int i = 0; i < CH; ++i)
                            if (it + g < steps && (m0 + (it + g) * SPW + sub) * L + q + LPS * i < D_left)
                                Elem<WT>::store(ptr + g * SPW * L + i * LPS, y[g][i]);
                }
                continue;
            }
#pragma unroll 8
            for (int it = 0; it < steps; ++it, ptr += SPW * L * VEC) {
                const int ms = it * SPW + sub;
                const float pm = __shfl_sync(kFull, p, ms);
                if (MODE != 0 && m0 + ms >= M_left) continue;
#pragma unroll
                for (int i = 0; i < CH; ++i) {
                    if constexpr (VEC == 1) {
                        if ((m0 + ms) * L + q + LPS * i < D_left) {
                            WT* pe = ptr + i * LPS;
                            float f = pm * vr[i][0];
                            if (beta) f += Elem<WT>::load(pe);
                            Elem<WT>::store(pe, f);
                        }
                        continue;
                    }
                    float y[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) y[e] = pm * vr[i][e % VEC];
                    if (MODE != 2) {
                        Out8<WT>::store(ptr + i * LPS * 8, y, beta);
                    } else {
                        const int col = ((m0 + ms) * L + q + LPS * i) * 8;
                        if (col + 8 <= D_left) {
                            Out8<WT>::store(ptr + i * LPS * 8, y, beta);
                        } else {
#pragma unroll
                            for (int e = 0; e < 8; ++e)
                                if (col + e < D_left) {
                                    WT* pe = ptr + i * LPS * 8 + e;
                                    float f = y[e];
                                    if (beta) f += Elem<WT>::load(pe);
                                    Elem<WT>::store(pe, f);
                                }
                        }
                    }
                }
            }
        }
    }
    }
}

template <int VEC, int LPS, int CH, typename ST, typename WT>
int launch_mode(int mode, int grid, const void* S, int splits, int64_t split_stride, int lds, const float* v,
                int R, int D, int M, int segs, int span, void* out, int64_t ldo, int beta, cudaStream_t stream)
{
    const ST* s = static_cast<const ST*>(S);
    WT* o = static_cast<WT*>(out);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid), 1, 1);
    cfg.blockDim = dim3(kStreamThreads, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr = pdl_attribute();
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaError_t e;
    if (mode == 0 && VEC == 8)
        e = cudaLaunchKernelEx(&cfg, expand_rows_vec_kernel<VEC, LPS, CH, VEC == 8 ? 0 : 2, ST, WT>, s, splits, split_stride, lds, v, R, D, M, segs, span, o, ldo, beta);
    else if (mode == 1 && VEC == 8)
        e = cudaLaunchKernelEx(&cfg, expand_rows_vec_kernel<VEC, LPS, CH, VEC == 8 ? 1 : 2, ST, WT>, s, splits, split_stride, lds, v, R, D, M, segs, span, o, ldo, beta);
    else
        e = cudaLaunchKernelEx(&cfg, expand_rows_vec_kernel<VEC, LPS, CH, 2, ST, WT>, s, splits, split_stride, lds, v, R, D, M, segs, span, o, ldo, beta);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return VELORA_ERR_CUDA;
    }
    return after_launch();
}

template <typename ST, typename WT>
int launch_shape(int vec, int lps, int ch, int mode, int grid, const void* S, int splits, int64_t split_stride, int lds,
                 const float* v, int R, int D, int M, int segs, int span, void* out, int64_t ldo, int beta, cudaStream_t stream)
{
#define VELORA_EXPAND_CASE(VECV, LPSV, CHV)                                                                    \
    if (vec == VECV && lps == LPSV && ch == CHV)                                                               \
        return launch_mode<VECV, LPSV, CHV, ST, WT>(mode, grid, S, splits, split_stride, lds, v, R, D, M, segs, span, out, ldo, beta, stream)
    VELORA_EXPAND_CASE(8, 1, 1);
    VELORA_EXPAND_CASE(8, 2, 1);
    VELORA_EXPAND_CASE(8, 4, 1);
    VELORA_EXPAND_CASE(8, 8, 1);
    VELORA_EXPAND_CASE(8, 16, 1);
    VELORA_EXPAND_CASE(8, 32, 1);
    VELORA_EXPAND_CASE(8, 32, 2);
    VELORA_EXPAND_CASE(8, 32, 4);
    VELORA_EXPAND_CASE(1, 8, 1);
    VELORA_EXPAND_CASE(1, 16, 1);
    VELORA_EXPAND_CASE(1, 32, 1);
    VELORA_EXPAND_CASE(1, 32, 2);
    VELORA_EXPAND_CASE(1, 32, 4);
    VELORA_EXPAND_CASE(1, 32, 8);
    VELORA_EXPAND_CASE(1, 32, 16);
    VELORA_EXPAND_CASE(1, 32, 32);
#undef VELORA_EXPAND_CASE
    return VELORA_ERR_UNSUPPORTED;
}

}  // namespace

int launch_expand_rows_vec(const void* S, int s_dtype, int splits, int64_t split_stride, int64_t lds, const float* v,
                           int64_t R, int64_t D, int Dsub, void* out, int out_dtype, int64_t ldo, int beta,
                           cudaStream_t stream)
{
    if (Dsub < 8 || Dsub > 1024 || (Dsub & (Dsub - 1))) return VELORA_ERR_UNSUPPORTED;
    const int vec = aligned16(out) && (ldo * static_cast<int64_t>(dtype_size(out_dtype))) % 16 == 0 ? 8 : 1;
    const int L = Dsub / vec;
    if (R < 1 || R >= (1 << 30) || lds >= (1 << 30) || D >= (1 << 30)) return VELORA_ERR_UNSUPPORTED;
    if ((s_dtype == VELORA_BF16 || s_dtype == VELORA_FP8_E4M3) && out_dtype != VELORA_BF16) return VELORA_ERR_UNSUPPORTED;
    const int lps = L < 32 ? L : 32, ch = L / lps;
    const int M = static_cast<int>(ceil_div64(D, Dsub));
    const int mode = (D % Dsub) ? 2 : ((M % 32) ? 1 : 0);
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc != VELORA_OK) return rc;
    const int64_t cap = static_cast<int64_t>(di.sm_count) * kStreamCtasPerSm, warps = cap * (kStreamThreads / 32);
    // Rows are cut while there are two warps and more for each, into spans of eight store instructions or more (four of 16 bytes).
    const int spw = 32 / lps, least = spw * ceil_div64(vec == 1 ? 8 : 4, ch);
    int64_t n_segs = R < warps ? warps / R : 1;
    if (n_segs > ceil_div64(M, least)) n_segs = ceil_div64(M, least);
    const int span = static_cast<int>(ceil_div64(ceil_div64(M, n_segs), spw) * spw);
    const int segs = static_cast<int>(ceil_div64(M, span));
    const int64_t ctas = ceil_div64(R * segs, kStreamThreads / 32);
    const int grid = static_cast<int>(ctas < cap ? ctas : cap);
    const int r = static_cast<int>(R), d = static_cast<int>(D), ld = static_cast<int>(lds);
    if (s_dtype == VELORA_BF16)
        return launch_shape<__nv_bfloat16, __nv_bfloat16>(vec, lps, ch, mode, grid, S, splits, split_stride, ld, v, r, d, M, segs, span, out, ldo, beta, stream);
    if (s_dtype == VELORA_FP8_E4M3)
        return launch_shape<e4m3_t, __nv_bfloat16>(vec, lps, ch, mode, grid, S, splits, split_stride, ld, v, r, d, M, segs, span, out, ldo, beta, stream);
    if (out_dtype == VELORA_BF16)
        return launch_shape<float, __nv_bfloat16>(vec, lps, ch, mode, grid, S, splits, split_stride, ld, v, r, d, M, segs, span, out, ldo, beta, stream);
    return launch_shape<float, float>(vec, lps, ch, mode, grid, S, splits, split_stride, ld, v, r, d, M, segs, span, out, ldo, beta, stream);
}

}  // namespace velora
