// Partial factors P[o, m] = sum_n dY[n, o] * Z[n, m] of token slices on the tensor cores, to fp32 accuracy, for the gradients that
// weight_grad_tc.cu does not take: fp32 rows, and bf16 rows on odd boundaries with Z as stored.
//
// An fp32 Z is split into three bf16 parts (exact, as in gemm_f32_tc.cu), the second and third side by side as columns of one operand: 64
// tokens of a bf16 dY are four tcgen05.mma of M = 128 columns of dY by N = round16(sub-tokens) and four by twice that.  An fp32 dY has three
// parts as well, and three times the products.  The tensor cores' sums truncate, so the products of the first parts, the only ones that
// reach the result's size, are added up there for 16 tokens and no further: 16 products of 16 significant bits hardly reach 24.
// The others share an accumulator for the 64 tokens of a stage, below 2^-7 of the result; after each stage all are read out
// and added to fp32 sums, rounded to nearest.
// Error in norm against 64 bits, 12608 x 768, 24 sub-tokens in fp32, this form / the 64 tokens in one accumulator / fp32
// multiply-adds on the CUDA cores, times 1e-8: |N(0, 1)| with a bf16 dY 4.7 / 8.9 / 4.8, fp32 4.1 / 7.1 / 4.8; N(0, 1) 9.9 / 11 / 17, 8.2 / 11 / 17.
//
// A CTA takes 128 columns of dY and one slice of the tokens.  Roles (416 threads): warps 0..3 sums (a lane has a column of dY);
// warps 4..11 operands (plain loads of any alignment, split, swizzled MN-major tiles: tokens are the contraction, rows of both
// matrices are rows of the tiles); warp 12 issues.  Two stages and two accumulators, a barrier pair each:
//   full[s] (eight operand warps), done[s] (commit: the stage may be written, the accumulator read), drained[a] (four warps).
// Two CTAs share an SM (bf16); bound by the loads and stores of the operand warps.  Rows that start on odd boundaries are
// read as the aligned 16 bytes that a chunk begins in and shifted against the neighbouring lane's.  Where the call has made a packed
// copy of dY for the input gradient already (TILED), a thirteenth warp fetches tiles of that instead, four stages deep, and the
// operand warps have Z only (layer of 4096 x 2048 -> 5461 with dense rows: 217 -> 203 us).
//
// Numbers that the parts cannot carry (split_bf16.cuh): the 32 columns of dY of a sum warp whose outputs may be wrong by what the operand
// warps have seen (in fp32 operands; how large a bf16 dY is they do not look at) or by what came out are computed by fp32 multiply-adds at
// the end.  12608 x 768 fp32, 24 sub-tokens: 21 us, 68 with every output computed again (32 on the CUDA cores).
#include "gemm_tc.cuh"
#include "row_chunks.cuh"
#include "split_bf16.cuh"
#include "tc_common.cuh"

namespace velora {

using namespace tc;

namespace {

constexpr int WP_O = 128, WP_K = 64;
constexpr int WP_SUM_WARPS = 4, WP_OPERAND_WARPS = 8;
constexpr int WP_OPERAND_THREADS = 32 * WP_OPERAND_WARPS;
constexpr int WP_THREADS = 32 * (WP_SUM_WARPS + WP_OPERAND_WARPS + 1);
constexpr int WP_FLAG_SHIFT = 16;                       // of the operands' flags in the word that says what to compute again
constexpr int WP_SLAB = WP_K * 128;                     // 64 columns of 64 tokens
constexpr int WP_A_PART = 2 * WP_SLAB;

template <typename YT, typename ZT, int MP, bool TILED>
struct PartsShape {
    static constexpr int kParts = sizeof(YT) == 2 ? 1 : 3;                      // of dY
    static constexpr int kZParts = sizeof(ZT) == 4 ? 3 : 1;                     // a stored bf16 or E4M3 value is a bf16 number
    static constexpr int kSlabsB = kZParts == 3 ? 2 : 1;                        // second and third parts of Z, then the first
    static constexpr int kHeadSlab = kSlabsB - 1;
    static constexpr int kStageBytes = kParts * WP_A_PART + kSlabsB * WP_SLAB;
    static constexpr int kStages = TILED ? (kStageBytes * 4 <= 100 * 1024 && MP == 16 ? 4 : 3) : 2;
    static constexpr int kThreads = WP_THREADS + (TILED ? 32 : 0);
    // What the roundings of the sums leave is kept beside them, in registers or, where those do not suffice, in shared memory.  An fp32 Z with
    // a bf16 dY does without: fp32 sums of its products on the CUDA cores were further off than this form is already.
    static constexpr bool kRests = kParts == 3 || kZParts == 1, kRestsInSmem = kParts == 1 && kRests && MP == 32;
    static constexpr size_t kSmem = 1024 + kStages * static_cast<size_t>(kStageBytes) + 128 + (kRestsInSmem ? WP_O * MP * 4 : 0);
    static constexpr int kCtasPerSm = kParts == 1 ? 2 : 1;
    // TMEM columns of a stage: first parts by first parts, four times 16 tokens; dY by the other parts of Z; the other parts of dY by the
    // first of Z.  Two such sets where the 512 columns of an SM have the room (not for a bf16 dY by an fp32 Z of more than 16 sub-tokens: 4096 x
    // 5461, 32 of them, 45 us instead of 42).
    static constexpr int kTailCol = (WP_K / 16) * MP, kSideCol = kTailCol + (kZParts == 3 ? 2 * MP : 0);
    static constexpr int kAccCols = kSideCol + (kParts == 3 ? MP : 0);
    static constexpr int kBuffers = 2 * kAccCols * kCtasPerSm <= 512 ? 2 : 1;
    static constexpr int kTmemCols = kBuffers * kAccCols <= 128 ? 128 : (kBuffers * kAccCols <= 256 ? 256 : 512);
    static_assert(kBuffers * kAccCols <= kTmemCols && kTmemCols * kCtasPerSm <= 512 && 2 * MP <= 64, "TMEM columns");
};

// dY of a stage: 64 tokens x 128 columns, four passes of sixteen tokens; a thread has eight columns of every sixteenth token.
template <typename YT> struct RowsOfY;

template <> struct RowsOfY<__nv_bfloat16> {
    uint4 x[4], over[4];
    __device__ __forceinline__ void load(const __nv_bfloat16* dY, int64_t ld, int n, int n_end, int o0, int, const char* end, int t)
    {
        const int l = t & 15;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int row = n + (t >> 4) + 16 * i;
            const char* rp = reinterpret_cast<const char*>(dY + static_cast<int64_t>(row) * ld + o0);
            const char* ap = rp - (reinterpret_cast<uintptr_t>(rp) & 15u) + 16 * l;
            x[i] = over[i] = make_uint4(0u, 0u, 0u, 0u);
            if (row < n_end) {
                x[i] = load_aligned_chunk(ap, reinterpret_cast<const char*>(dY), end);
                if (l == 15) over[i] = load_aligned_chunk(ap + 16, reinterpret_cast<const char*>(dY), end);
            }
        }
    }
    __device__ __forceinline__ void store(uint32_t a0, const __nv_bfloat16* dY, int64_t ld, int n, int o0, int t, SplitOperandCheck&)
    {
        const int r = t >> 4, l = t & 15;
        const uint32_t at = a0 + (l >> 3) * WP_SLAB + r * 128 + (((l & 7) ^ (r & 7)) << 4);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t shift = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(dY + static_cast<int64_t>(n + r + 16 * i) * ld + o0) & 15u);
            uint4 y;
            y.x = __shfl_down_sync(0xffffffffu, x[i].x, 1, 16); y.y = __shfl_down_sync(0xffffffffu, x[i].y, 1, 16);
            y.z = __shfl_down_sync(0xffffffffu, x[i].z, 1, 16); y.w = __shfl_down_sync(0xffffffffu, x[i].w, 1, 16);
            const uint4 w = shift_chunks(x[i], l == 15 ? over[i] : y, shift);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at + i * 16 * 128), "r"(w.x), "r"(w.y), "r"(w.z), "r"(w.w) : "memory");
        }
    }
};

template <> struct RowsOfY<float> {
    float4 x[8];                                       // eight tokens a pass: four columns of every eighth token
    __device__ __forceinline__ void load(const float* dY, int64_t ld, int n, int n_end, int o0, int O, const char*, int t)
    {
        const int c = (t & 31) * 4, left = O - (o0 + c);
        const bool vec = (reinterpret_cast<uintptr_t>(dY) & 15u) == 0 && ld % 4 == 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int row = n + (t >> 5) + 8 * i;
            const float* q = dY + static_cast<int64_t>(row) * ld + o0 + c;
            x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row >= n_end) continue;
            if (vec && left >= 4) {
                x[i] = *reinterpret_cast<const float4*>(q);
            } else {
                if (left > 0) x[i].x = q[0];
                if (left > 1) x[i].y = q[1];
                if (left > 2) x[i].z = q[2];
                if (left > 3) x[i].w = q[3];
            }
        }
    }
    __device__ __forceinline__ void store(uint32_t a0, const float*, int64_t, int, int, int t, SplitOperandCheck& seen)
    {
        const int r = t >> 5, c = (t & 31) * 4;
        const uint32_t at = a0 + (c >> 6) * WP_SLAB + r * 128 + ((((c >> 3) & 7) ^ r) << 4) + (c & 4) * 2;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float2 a = make_float2(x[i].x, x[i].y), b = make_float2(x[i].z, x[i].w);
            seen.add(a);
            seen.add(b);
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                if (p == 2) {
                    seen.add_rest(a);
                    seen.add_rest(b);
                }
                const uint32_t u = pack_bf16x2(a.x, a.y), w = pack_bf16x2(b.x, b.y);
                asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at + i * 8 * 128 + p * WP_A_PART), "r"(u), "r"(w) : "memory");
                if (p < 2) {
                    a = minus_parts(a, u);
                    b = minus_parts(b, w);
                }
            }
        }
    }
};

// Z of a stage: 64 tokens x MP sub-tokens (zeros beyond M and n_end), a thread has pairs of neighbours.
template <typename YT, typename ZT, int MP>
struct RowsOfZ {
    static constexpr int kPairs = WP_K * MP / 2 / WP_OPERAND_THREADS;
    float2 x[kPairs];
    __device__ __forceinline__ void load(const ZT* Z, int64_t ld, int n, int n_end, int M, int t)
    {
#pragma unroll
        for (int i = 0; i < kPairs; ++i) {
            const int idx = t + WP_OPERAND_THREADS * i, row = n + idx / (MP / 2), m = idx % (MP / 2) * 2;
            const ZT* q = Z + static_cast<int64_t>(row) * ld + m;
            x[i].x = row < n_end && m < M ? Elem<ZT>::load(q) : 0.f;
            x[i].y = row < n_end && m + 1 < M ? Elem<ZT>::load(q + 1) : 0.f;
        }
    }
    __device__ __forceinline__ void store(uint32_t b0, int t, SplitOperandCheck& seen)
    {
#pragma unroll
        for (int i = 0; i < kPairs; ++i) {
            const int idx = t + WP_OPERAND_THREADS * i, r = idx / (MP / 2), m = idx % (MP / 2) * 2;
            float2 a = x[i];
            if (sizeof(YT) == 4) seen.add(a);
#pragma unroll
            for (int p = 0; p < (sizeof(ZT) == 4 ? 3 : 1); ++p) {
                if (p == 2) seen.add_rest(a);                        // columns beyond M and rows beyond n_end are zeros
                const int c = p == 0 ? m : (p - 1) * MP + m;
                const uint32_t u = pack_bf16x2(a.x, a.y);
                asm volatile("st.shared.b32 [%0], %1;"
                             ::"r"(b0 + (p == 0 && sizeof(ZT) == 4 ? WP_SLAB : 0) + r * 128 + (((c >> 3) ^ (r & 7)) << 4) + (c & 7) * 2), "r"(u) : "memory");
                if (p < 2 && sizeof(ZT) == 4) a = minus_parts(a, u);
            }
        }
    }
};

// The marked outputs (bit w: those of sum warp w) by fp32 multiply-adds, whole CTA: warps 0 .. 11 have 32 columns of dY by 8 sub-tokens
// each, 64 tokens of Z at a time in shared memory (`zs`, 64 x 24) and added to the sum.
template <typename YT, typename ZT>
__device__ __noinline__ void redo_outputs(const YT* dY, int64_t lddy, const ZT* Z, int64_t ldz, int n_begin, int n_end, int o0, int O, int M,
                                          uint32_t marked, float* zs, float* out)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, block = warp & 3, third = warp >> 2;
    const int o = o0 + block * 32 + lane;
    const YT* y = dY + (o < O ? o : O - 1);
    for (int m_first = 0; m_first < M; m_first += 24) {
        const int m0 = m_first + 8 * third;
        const bool mine = third < 3 && m0 < M && ((marked >> block) & 1u);
        float sum[8] = {};
        for (int n0 = n_begin; n0 < n_end; n0 += WP_K) {
            __syncthreads();
            for (int i = threadIdx.x; i < WP_K * 24; i += blockDim.x) {
                const int n = n0 + i / 24, m = m_first + i % 24;
                zs[i] = n < n_end && m < M ? Elem<ZT>::load(Z + static_cast<int64_t>(n) * ldz + m) : 0.f;
            }
            __syncthreads();
            if (!mine) continue;
            float part[8] = {};
#pragma unroll 1
            for (int h = 0; h < WP_K; h += 16) {
                float f[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) f[i] = n0 + h + i < n_end ? Elem<YT>::load(y + static_cast<int64_t>(n0 + h + i) * lddy) : 0.f;
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float4 u = *reinterpret_cast<const float4*>(zs + (h + i) * 24 + 8 * third), w = *reinterpret_cast<const float4*>(zs + (h + i) * 24 + 8 * third + 4);
                    part[0] = fmaf(f[i], u.x, part[0]); part[1] = fmaf(f[i], u.y, part[1]);
                    part[2] = fmaf(f[i], u.z, part[2]); part[3] = fmaf(f[i], u.w, part[3]);
                    part[4] = fmaf(f[i], w.x, part[4]); part[5] = fmaf(f[i], w.y, part[5]);
                    part[6] = fmaf(f[i], w.z, part[6]); part[7] = fmaf(f[i], w.w, part[7]);
                }
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) sum[e] += part[e];
        }
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (mine && o < O && m0 + e < M) out[static_cast<int64_t>(o) * M + m0 + e] = sum[e];
    }
}

template <typename YT, typename ZT, int MP, bool TILED>
__global__ void __launch_bounds__(PartsShape<YT, ZT, MP, TILED>::kThreads, PartsShape<YT, ZT, MP, TILED>::kCtasPerSm)
wg_parts_kernel(const __grid_constant__ CUtensorMap tmY, const YT* dY, int64_t lddy, const ZT* Z, int64_t ldz, int N, int O, int M, int tokens_per_cta,
                float* __restrict__ partials, int* __restrict__ status)
{
    using S = PartsShape<YT, ZT, MP, TILED>;
    constexpr uint32_t ST = S::kStages;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* tail = smem_raw + (base - raw) + ST * S::kStageBytes;
    const uint32_t full = base + ST * S::kStageBytes, done = full + 32, drained = full + 64;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tail + 80);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 88);
    uint32_t* redo = reinterpret_cast<uint32_t*>(tail + 92);              // bit w: the columns of sum warp w
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int o0 = blockIdx.y * WP_O;
    const int n_begin = blockIdx.x * tokens_per_cta;
    const int n_end = n_begin + tokens_per_cta < N ? n_begin + tokens_per_cta : N;

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < ST; ++s) {
            mbar_init(full + 8 * s, WP_OPERAND_WARPS + (TILED ? 1 : 0));
            mbar_init(done + 8 * s, 1);
        }
        for (int a = 0; a < 2; ++a) mbar_init(drained + 8 * a, WP_SUM_WARPS);
        if (TILED) prefetch_tensormap(&tmY);
        *abort_flag = 0;
        *redo = 0;
        fence_mbar_init();
    }
    if (warp == WP_SUM_WARPS + WP_OPERAND_WARPS) {
        tmem_alloc(smem_u32(tmem_slot), S::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;

    bool failed = false;
    if (TILED && warp > WP_SUM_WARPS + WP_OPERAND_WARPS) {
        // ------------------------------------------------ tiles of the packed copy of dY
        if (lane == 0) {
            uint32_t it = 0;
            for (int n = n_begin; n < n_end; n += WP_K, ++it) {
                const uint32_t s = it % ST, ph = (it / ST) & 1u;
                if (!mbar_wait(done + 8 * s, ph ^ 1u, abort_flag)) { failed = true; break; }
                mbar_arrive_expect_tx(full + 8 * s, WP_A_PART);
                tma_load_2d(base + s * S::kStageBytes, &tmY, full + 8 * s, o0, n);
                tma_load_2d(base + s * S::kStageBytes + WP_SLAB, &tmY, full + 8 * s, o0 + 64, n);
            }
            if (failed) {
                *abort_flag = 1;
                // The copies in flight land before shared memory is given up; their stages may lack other arrivals, so by the clock.
                const unsigned long long t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 50000ull) __nanosleep(1000);
            }
        }
    } else if (warp == WP_SUM_WARPS + WP_OPERAND_WARPS) {
        // ------------------------------------------------ products
        if (lane == 0) {
            constexpr uint32_t idesc_head = umma_idesc_bf16(WP_O, MP, true, true), idesc_tail = umma_idesc_bf16(WP_O, 2 * MP, true, true);
            uint32_t it = 0;
            for (int n = n_begin; n < n_end; n += WP_K, ++it) {
                const uint32_t s = it % ST, ph = (it / ST) & 1u, acc = it % S::kBuffers;
                if (!mbar_wait(drained + 8 * acc, ((it / S::kBuffers) & 1u) ^ 1u, abort_flag) || !mbar_wait(full + 8 * s, ph, abort_flag)) { failed = true; break; }
                tc_fence_after_sync();
                const uint32_t a0 = base + s * S::kStageBytes, b0 = a0 + S::kParts * WP_A_PART, d = tmem_base + acc * S::kAccCols;
#pragma unroll
                for (int p = S::kParts - 1; p >= 0; --p)
#pragma unroll
                    for (int j = 0; j < WP_K / 16; ++j) {
                        const bool more = p != S::kParts - 1 || j != 0;
                        const uint64_t a = umma_smem_desc(a0 + p * WP_A_PART + j * 2048, WP_SLAB, 1024);
                        if (S::kZParts == 3) umma_bf16(d + S::kTailCol, a, umma_smem_desc(b0 + j * 2048, WP_SLAB, 1024), idesc_tail, more);
                        umma_bf16(d + (p == 0 ? j * MP : S::kSideCol), a, umma_smem_desc(b0 + S::kHeadSlab * WP_SLAB + j * 2048, WP_SLAB, 1024), idesc_head,
                                  p != 0 && more);
                    }
                umma_commit(done + 8 * s);
            }
            if (failed) *abort_flag = 1;
        }
    } else if (warp >= WP_SUM_WARPS) {
        // ------------------------------------------------ operands
        const int t = threadIdx.x - 32 * WP_SUM_WARPS;
        const char* end = reinterpret_cast<const char*>(dY + static_cast<int64_t>(N - 1) * lddy + O);
        RowsOfY<YT> y;
        RowsOfZ<YT, ZT, MP> z;
        SplitOperandCheck seen;
        if (!TILED) y.load(dY, lddy, n_begin, n_end, o0, O, end, t);
        z.load(Z, ldz, n_begin, n_end, M, t);
        uint32_t it = 0;
        for (int n = n_begin; n < n_end; n += WP_K, ++it) {
            const uint32_t s = it % ST, ph = (it / ST) & 1u;
            if (!mbar_wait_warp(done + 8 * s, ph ^ 1u, abort_flag)) { failed = true; break; }
            const uint32_t a0 = base + s * S::kStageBytes;
            if (!TILED) y.store(a0, dY, lddy, n, o0, t, seen);
            z.store(a0 + S::kParts * WP_A_PART, t, seen);
            if (n + WP_K >= n_end && seen.flags()) atomicOr(redo, (sizeof(YT) == 2 ? SPLIT_TINY | SPLIT_BIG : seen.flags()) << WP_FLAG_SHIFT);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(full + 8 * s);
            if (n + WP_K < n_end) {
                if (!TILED) y.load(dY, lddy, n + WP_K, n_end, o0, O, end, t);
                z.load(Z, ldz, n + WP_K, n_end, M, t);
            }
        }
        if (failed) *abort_flag = 1;
    } else {
        // ------------------------------------------------ sums: lane = column o of dY
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(warp * 32) << 16);
        float sum[MP], rest[MP];
        float* shared_rest = reinterpret_cast<float*>(tail + 128) + threadIdx.x;
#pragma unroll
        for (int m = 0; m < MP; ++m) {
            sum[m] = rest[m] = 0.f;
            if (S::kRestsInSmem) shared_rest[m * WP_O] = 0.f;
        }
        uint32_t it = 0;
        for (int n = n_begin; n < n_end; n += WP_K, ++it) {
            const uint32_t s = it % ST, ph = (it / ST) & 1u, acc = it % S::kBuffers;
            if (!mbar_wait_warp(done + 8 * s, ph, abort_flag, 32)) { failed = true; break; }
            tc_fence_after_sync();
#pragma unroll
            for (int m = 0; m < MP; m += 8) {                        // what a stage brings first, then one rounding of the sum
                const uint32_t at = taddr + acc * S::kAccCols + m;
                float head[8];
#pragma unroll
                for (int j = 0; j < WP_K / 16; j += 2) {
                    uint32_t x[8], y[8];
                    tmem_ld_32x8(at + j * MP, x);
                    tmem_ld_32x8(at + (j + 1) * MP, y);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const float f = __uint_as_float(x[e]) + __uint_as_float(y[e]);
                        head[e] = j == 0 ? f : head[e] + f;
                    }
                }
                if (S::kAccCols > S::kTailCol) {
                    uint32_t mid[8] = {}, l[8] = {}, side[8] = {};
                    if (S::kZParts == 3) {
                        tmem_ld_32x8(at + S::kTailCol, mid);
                        tmem_ld_32x8(at + S::kTailCol + MP, l);
                    }
                    if (S::kParts == 3) tmem_ld_32x8(at + S::kSideCol, side);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        float f = S::kZParts == 3 ? __uint_as_float(mid[e]) + __uint_as_float(l[e]) : 0.f;
                        if (S::kParts == 3) f += __uint_as_float(side[e]);
                        head[e] += f;
                    }
                }
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    if (S::kRests) {
                        const float next = sum[m + e] + head[e];
                        (S::kRestsInSmem ? shared_rest[(m + e) * WP_O] : rest[m + e]) += head[e] - (next - sum[m + e]);
                        sum[m + e] = next;
                    } else {
                        sum[m + e] += head[e];
                    }
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(drained + 8 * acc);
        }
        const int o = o0 + warp * 32 + lane;
        float* out = partials + (static_cast<int64_t>(blockIdx.x) * O + o) * M;
        SplitOutputCheck check;
#pragma unroll
        for (int m = 0; m < MP; ++m) {
            if (S::kRests) sum[m] += S::kRestsInSmem ? shared_rest[m * WP_O] : rest[m];
            if (o < O && m < M) {
                out[m] = sum[m];
                check.add(sum[m]);
            }
        }
        const uint32_t operands = *const_cast<volatile uint32_t*>(redo) >> WP_FLAG_SHIFT;
        if (check.suspect(operands, n_end - n_begin)) atomicOr(redo, 1u << warp);
        if (failed) *abort_flag = 1;
    }
    if (failed && status) atomicExch(status, VELORA_ERR_TIMEOUT);

    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == WP_SUM_WARPS + WP_OPERAND_WARPS) {
        __syncwarp();
        tmem_dealloc(tmem_base, S::kTmemCols);
    }
    if ((*redo & 0xfu) && !*abort_flag)
        redo_outputs<YT, ZT>(dY, lddy, Z, ldz, n_begin, n_end, o0, O, M, *redo, reinterpret_cast<float*>(smem_raw + (base - raw)),
                             partials + static_cast<int64_t>(blockIdx.x) * O * M);
}

struct PartsArgs {
    const void *dY, *Z;
    int64_t lddy, ldz;
    int N, O, M, tokens_per_cta, parts;
    float* partials;
    int* status;
};

template <typename YT, typename ZT, int MP, bool TILED>
int launch_shape(const CUtensorMap& tmY, const PartsArgs& a, cudaStream_t stream)
{
    using S = PartsShape<YT, ZT, MP, TILED>;
    static DeviceOnce configured;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return VELORA_ERR_CUDA;
    auto kern = wg_parts_kernel<YT, ZT, MP, TILED>;
    if (!configured.get(dev)) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(S::kSmem)) != cudaSuccess) return VELORA_ERR_CUDA;
        configured.set(dev);
    }
    const dim3 grid(static_cast<unsigned>(a.parts), static_cast<unsigned>(ceil_div64(a.O, WP_O)));
    kern<<<grid, S::kThreads, S::kSmem, stream>>>(tmY, static_cast<const YT*>(a.dY), a.lddy, static_cast<const ZT*>(a.Z), a.ldz, a.N, a.O, a.M,
                                                  a.tokens_per_cta, a.partials, a.status);
    return after_launch();
}

template <typename YT, typename ZT>
int launch_types(const PartsArgs& a, const void* packed, int64_t ld_packed, cudaStream_t stream)
{
    CUtensorMap tm = {};
    if (sizeof(YT) == 2 && packed && make_tmap_bf16_2d(&tm, packed, a.O, a.N, ld_packed, 64, WP_K) == VELORA_OK)
        return a.M <= 16 ? launch_shape<__nv_bfloat16, ZT, 16, true>(tm, a, stream) : launch_shape<__nv_bfloat16, ZT, 32, true>(tm, a, stream);
    return a.M <= 16 ? launch_shape<YT, ZT, 16, false>(tm, a, stream) : launch_shape<YT, ZT, 32, false>(tm, a, stream);
}

}  // namespace

int wg_parts_slices(int dy_dtype, int64_t O, int sm_count)
{
    const int64_t slices = static_cast<int64_t>(sm_count) * (dy_dtype == VELORA_BF16 ? 2 : 1) / ceil_div64(O, WP_O);
    return slices < 1 ? 1 : static_cast<int>(slices);
}

int launch_wg_parts(const void* dY, int dy_dtype, int64_t lddy, const void* packed, int64_t ld_packed, const void* Z, int z_dtype, int64_t ldz,
                    int N, int O, int M, int tokens_per_cta, int parts, float* partials, int* status, cudaStream_t stream)
{
    const PartsArgs a{dY, Z, lddy, ldz, N, O, M, tokens_per_cta, parts, partials, status};
#define VELORA_WP_CASE(YT)                                                                                     \
    if (z_dtype == VELORA_FP8_E4M3) return launch_types<YT, e4m3_t>(a, packed, ld_packed, stream);             \
    if (z_dtype == VELORA_BF16) return launch_types<YT, __nv_bfloat16>(a, packed, ld_packed, stream);          \
    return launch_types<YT, float>(a, packed, ld_packed, stream)
    if (dy_dtype == VELORA_BF16) { VELORA_WP_CASE(__nv_bfloat16); }
    VELORA_WP_CASE(float);
#undef VELORA_WP_CASE
}

}  // namespace velora
