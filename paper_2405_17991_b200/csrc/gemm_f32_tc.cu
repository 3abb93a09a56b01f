// Dense products of Algorithm 1 (arxiv 2405.17991) for fp32 operands on the tensor cores, to fp32 accuracy:
//   C[m, n] = beta * C[m, n] + sum_k A(m, k) * B(n, k)
//
// Every fp32 number is the sum of three bf16 numbers, x = h + m + l, exactly (8 + 8 + 8 significant bits), so a product is six
// bf16 products (h h', h m', m h', m m', h l', l h') and a remainder below 2^-26 of it.  A k-block of 64 is staged as
// three bf16 tiles per operand and multiplied six times, the small products first.  The tensor cores add with truncation, so
// their sum is not left to grow: after every k-block the accumulator is read out and added, rounded to nearest, to sums in
// registers.  Error in norm against 64 bits, 2048 x 2048 outputs, this form / fp32 multiply-adds in sequence:
//   K = 64: 0.8e-7 / 1.4e-7,  K = 768: 1.0e-7 / 5.0e-7,  K = 3072: 1.5e-7 / 9.9e-7
// (accumulators read out every 128 instead of every 64: 5.9e-7 at any K), and on |N(0, 1)|, whose products are all of one sign,
//   K = 64: 0.9e-7 / 1.2e-7,  K = 768: 1.0e-7 / 3.7e-7,  K = 3072: 1.3e-7 / 7.4e-7.
//
// CTA pairs (cta_group::2), 256 x BN outputs a pair, BN = 192 (or 96).  12608 x 768, K = 768: 97 us, 153 TFLOP/s of fp32 arithmetic
// (372 us on the CUDA cores).  Nearest to a limit by count is shared memory: a k-block's 24 products read 172 KB of operands, the
// split writes 86 KB and its loads pass 114 KB through, 2900 cycles of 128 bytes where the tensor cores need 2310; the block takes
// 3400 (over the whole launch the tensor pipe is busy for 51 % of the cycles, the schedulers issue in 52 %).  Registers decide the split of roles: 12 warps of sums with 64 columns each, so few registers for the operand warps that
// only A of the next k-block waits in them (both operands, and spills: 115 us; eight operand warps: 101).
//
// Roles per CTA (1024 threads):
//   warps 0..11   sums: warp w has TMEM lanes 32 * (w % 4) .. and a third of the columns, BN / 3 registers a thread.  They
//                 write C, while the products of the next tile are already running.
//   warps 12..27  operands: read the k-block after the one being multiplied from global memory into registers, split it and
//                 write the tiles (128-byte swizzle, K-major or MN-major like the source: nothing is transposed).
//   warps 28, 29  leader: 28 issues the products of both CTAs.  Peer: they pass its full and drained barriers on to the leader's
//                 (30, 31 idle: registers are shared out by four warps).
// Barriers, two of each (a k-block has a stage and an accumulator):
//   full[s]       one per CTA, the operand warps; the leader's also has the peer's.
//   done[s]       one per CTA (multicast commit): the stage may be refilled, the accumulator may be read.
//   drained[s]    one per CTA, the sum warps; the leader's also has the peer's.
// An arrival on the other CTA's barrier holds its warp up for 700 to 1000 cycles, which the operand and sum warps do not have.
// Every wait is bounded; both CTAs always reach the closing cluster barrier.  No copies are in flight when they do.
//
// Numbers that the split cannot carry (split_bf16.cuh).  The operand warps look at what they split and leave a tile's flags in its word of
// marks, in both CTAs, before its last full[s]; a warp whose 32 x BN / 3 outputs may be wrong by them or by what came out leaves the outputs
// unwritten and sets its bit there.  Marked outputs are computed by fp32 multiply-adds behind the last tile, when no role waits for
// another any more (computed in between they kept the pair's other roles waiting, for longer than those do when a contraction is long), at
// about the rate of the CUDA-core product: 12608 x 768 x 768 with every output marked 640 us, with one row 229.
#include <cooperative_groups.h>

#include <type_traits>

#include "gemm_store.cuh"
#include "gemm_tc.cuh"
#include "split_bf16.cuh"
#include "tc_pair.cuh"

namespace velora {

using namespace tc;

namespace {

constexpr int F_BM = 128;                          // rows per CTA
constexpr int F_BK = 64;
constexpr int F_SUM_WARPS = 12, F_OPERAND_WARPS = 16;
constexpr int F_OPERAND_THREADS = 32 * F_OPERAND_WARPS;
constexpr int F_THREADS = 32 * (F_SUM_WARPS + F_OPERAND_WARPS + 4);
// Registers a thread: launched with 64, then shared out by warpgroups (12 + 16 + 4 warps), in total what the launch has.
constexpr int F_SUM_REGS = 88, F_OPERAND_REGS = 48, F_ISSUE_REGS = 48;
static_assert(F_SUM_WARPS * F_SUM_REGS + F_OPERAND_WARPS * F_OPERAND_REGS + 4 * F_ISSUE_REGS <= F_THREADS / 32 * 64, "registers of the launch");
constexpr int F_SLAB = 64 * F_BK * 2;              // 64 columns of an MN-major tile
constexpr int F_STAGES = 2;                        // stage = accumulator = k-block mod 2
constexpr int F_STAGE_PITCH = 17;                  // 16 columns of 32 unaligned output rows, no bank conflicts either way
constexpr int F_BARRIER_BYTES = 128;
constexpr int F_FLAG_SHIFT = 16;                   // of the operands' flags in a tile's word of marks

template <int N> using Int = std::integral_constant<int, N>;

struct F32Operand {
    const float* p;
    int64_t ld;                                    // pitch of the contiguous rows in memory
    int vec;                                       // whether they start on 16-byte boundaries
};

// Four elements of a row, of which `left` exist; zeros for the others.
__device__ __forceinline__ float4 load4(const float* q, int left, int vec)
{
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (vec && left >= 4) {
        x = __ldg(reinterpret_cast<const float4*>(q));
    } else {
        if (left > 0) x.x = __ldg(q);
        if (left > 1) x.y = __ldg(q + 1);
        if (left > 2) x.z = __ldg(q + 2);
        if (left > 3) x.w = __ldg(q + 3);
    }
    return x;
}

// One operand's tile of a k-block: W of its rows m (or n) times 64 of k.  `MN`: memory is contiguous along m (or n).  A thread
// has four consecutive elements of every kRowsPerPass-th row.
template <bool MN, int W>
struct SplitTile {
    static constexpr int kCols = MN ? W : F_BK;                       // contiguous in memory and in the tile
    static constexpr int kRows = MN ? F_BK : W;
    static constexpr int kLanes = kCols > 64 ? 32 : 16;               // threads along a row
    static constexpr int kRowsPerPass = F_OPERAND_THREADS / kLanes;   // a multiple of 8: the swizzle is the same in every pass
    static constexpr int kPasses = (kRows + kRowsPerPass - 1) / kRowsPerPass;
    static constexpr int kPartBytes = (MN ? (W + 63) / 64 * F_SLAB : W * F_BK * 2);
    static_assert(kCols <= 4 * kLanes && kRowsPerPass % 8 == 0 && kPartBytes % 1024 == 0 && kPasses <= 4, "tile shape");

    const float* q;                               // this thread's first element of the k-block
    int rows, cols;                               // how many rows and elements of a row there are from it on

    __device__ __forceinline__ void start(const F32Operand& op, int mn0, int mn, int k, int t)      // k-block 0 of a tile that begins at mn0
    {
        const int r = t / kLanes, c = t % kLanes * 4;
        q = op.p + static_cast<int64_t>(MN ? r : mn0 + r) * op.ld + (MN ? mn0 + c : c);
        rows = (MN ? k : min(mn - mn0, W)) - r;
        cols = c < kCols ? (MN ? mn - mn0 : k) - c : 0;
    }
    __device__ __forceinline__ void advance(const F32Operand& op)
    {
        q += MN ? F_BK * op.ld : F_BK;
        if (MN) rows -= F_BK;
        else cols -= F_BK;
    }
    __device__ __forceinline__ float4 load(const F32Operand& op, int pass) const
    {
        return load4(q + pass * (kRowsPerPass * op.ld), pass * kRowsPerPass < rows ? cols : 0, op.vec);
    }
    // The three parts, kPartBytes apart.
    static __device__ __forceinline__ void store(uint32_t part0, int pass, int t, const float4& x, SplitOperandCheck& seen)
    {
        const int r = t / kLanes, c = t % kLanes * 4;
        if (c >= kCols || (kRows % kRowsPerPass && r + pass * kRowsPerPass >= kRows)) return;
        const uint32_t at = part0 + (c >> 6) * F_SLAB + r * 128 + ((((c >> 3) & 7) ^ (r & 7)) << 4) + (c & 4) * 2 + pass * (kRowsPerPass * 128);
        float2 a = make_float2(x.x, x.y), b = make_float2(x.z, x.w);
        seen.add(a);
        seen.add(b);
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            if (p == 2) {
                seen.add_rest(a);
                seen.add_rest(b);
            }
            const uint32_t u = pack_bf16x2(a.x, a.y), w = pack_bf16x2(b.x, b.y);
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at + p * kPartBytes), "r"(u), "r"(w) : "memory");
            if (p < 2) {
                a = minus_parts(a, u);
                b = minus_parts(b, w);
            }
        }
    }
};

template <bool A_MN, bool B_MN, int BN>
struct F32Shape {
    using TileA = SplitTile<A_MN, F_BM>;
    using TileB = SplitTile<B_MN, BN / 2>;
    static constexpr int kStageBytes = 3 * (TileA::kPartBytes + TileB::kPartBytes);
    static constexpr int kAccCols = BN > 128 ? 256 : 128;             // TMEM columns from one accumulator to the next
    static constexpr int kMaxTiles = BN > 128 ? 2048 : 1024;          // of a pair in one launch, one word of marks each
    static constexpr size_t kSmem = 1024 + static_cast<size_t>(F_STAGES) * kStageBytes + F_BARRIER_BYTES +
                                    F_SUM_WARPS * 32 * F_STAGE_PITCH * sizeof(float) + kMaxTiles * sizeof(uint32_t);
};

__device__ __forceinline__ void sum_warps_sync() { asm volatile("bar.sync 1, %0;" ::"n"(32 * F_SUM_WARPS) : "memory"); }
// The same; true in all of them if `p` is in one.
__device__ __forceinline__ bool sum_warps_any(bool p)
{
    uint32_t any;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(any) : "r"(static_cast<uint32_t>(p)), "n"(32 * F_SUM_WARPS) : "memory");
    return any != 0;
}

// Sets bits of a word of shared memory in both CTAs of the pair, before any arrival that this thread makes afterwards.
__device__ __noinline__ void flag_tile(uint32_t* word, uint32_t bits)
{
    const uint32_t local = smem_u32(word);
    for (uint32_t rank = 0; rank < 2; ++rank)
        asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(map_to_cta(local, rank)), "r"(bits) : "memory");
    asm volatile("fence.acq_rel.cluster;" ::: "memory");
}

// Four bytes to shared memory, zero where `take` is false.
__device__ __forceinline__ void copy4_async(uint32_t dst, const float* src, bool take)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(take ? 4 : 0) : "memory");
}

// The marked outputs of a CTA's 128 x BN (bit w: those of sum warp w) by fp32 multiply-adds, all sum warps: blocks of 96 columns, 8 x 4
// outputs a thread, slices of 32 through the ring's memory, the next one on its way while one is multiplied.
constexpr int F_REDO_COLS = 96, F_REDO_K = 32, F_REDO_PITCH_A = F_BM + 4, F_REDO_PITCH_B = F_REDO_COLS + 4;
constexpr int F_REDO_SLICE = F_REDO_K * (F_REDO_PITCH_A + F_REDO_PITCH_B);          // floats

template <bool A_MN, bool B_MN>
__device__ __forceinline__ void redo_load(const F32Operand& A, const F32Operand& B, int m0, int n0, int k0, int Mdim, int Ndim, int Kdim,
                                          uint32_t slice, int t)
{
#pragma unroll 4
    for (int i = t; i < F_BM * F_REDO_K; i += 32 * F_SUM_WARPS) {
        const int r = A_MN ? i % F_BM : i / F_REDO_K, k = A_MN ? i / F_BM : i % F_REDO_K, m = m0 + r;
        const bool in = m < Mdim && k0 + k < Kdim;
        const float* q = A.p + (A_MN ? static_cast<int64_t>(k0 + k) * A.ld + m : static_cast<int64_t>(m) * A.ld + (k0 + k));
        copy4_async(slice + (k * F_REDO_PITCH_A + r) * 4, in ? q : A.p, in);
    }
#pragma unroll 4
    for (int i = t; i < F_REDO_COLS * F_REDO_K; i += 32 * F_SUM_WARPS) {
        const int c = B_MN ? i % F_REDO_COLS : i / F_REDO_K, k = B_MN ? i / F_REDO_COLS : i % F_REDO_K, n = n0 + c;
        const bool in = n < Ndim && k0 + k < Kdim;
        const float* q = B.p + (B_MN ? static_cast<int64_t>(k0 + k) * B.ld + n : static_cast<int64_t>(n) * B.ld + (k0 + k));
        copy4_async(slice + (F_REDO_K * F_REDO_PITCH_A + k * F_REDO_PITCH_B + c) * 4, in ? q : B.p, in);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

template <bool A_MN, bool B_MN, int BN>
__device__ __noinline__ void redo_tile(const F32Operand A, const F32Operand B, float* C, int64_t ldc, int beta, int m0, int n0,
                                       int Mdim, int Ndim, int Kdim, uint32_t marked, float* ring)
{
    static_assert(F_SUM_WARPS * 32 == F_BM / 8 * (F_REDO_COLS / 4) && BN % F_REDO_COLS == 0, "one block at a time");
    const int t = threadIdx.x, tr = t / (F_REDO_COLS / 4) * 8, tc = t % (F_REDO_COLS / 4) * 4;
    for (int u0 = 0; u0 < BN && n0 + u0 < Ndim; u0 += F_REDO_COLS) {
        // Eight rows of a thread are within a warp's 32, four columns within its third.
        const bool mine = (marked >> ((u0 + tc) / (BN / 3) * 4 + tr / 32)) & 1u, work = __any_sync(0xffffffffu, mine);
        float acc[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
        sum_warps_sync();                                   // the last block's slices have been read
        redo_load<A_MN, B_MN>(A, B, m0, n0 + u0, 0, Mdim, Ndim, Kdim, smem_u32(ring), t);
        int odd = 0;
        for (int k0 = 0; k0 < Kdim; k0 += F_REDO_K, odd ^= 1) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            sum_warps_sync();                               // this slice is there, the one before it has been read
            if (k0 + F_REDO_K < Kdim)
                redo_load<A_MN, B_MN>(A, B, m0, n0 + u0, k0 + F_REDO_K, Mdim, Ndim, Kdim, smem_u32(ring + (odd ^ 1) * F_REDO_SLICE), t);
            if (!work) continue;
            const float* sA = ring + odd * F_REDO_SLICE + tr;
            const float* sB = ring + odd * F_REDO_SLICE + F_REDO_K * F_REDO_PITCH_A + tc;
#pragma unroll 4
            for (int k = 0; k < F_REDO_K; ++k) {
                const float4 a0 = *reinterpret_cast<const float4*>(sA + k * F_REDO_PITCH_A), a1 = *reinterpret_cast<const float4*>(sA + k * F_REDO_PITCH_A + 4);
                const float4 b = *reinterpret_cast<const float4*>(sB + k * F_REDO_PITCH_B);
                const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    acc[i][0] = fmaf(a[i], b.x, acc[i][0]);
                    acc[i][1] = fmaf(a[i], b.y, acc[i][1]);
                    acc[i][2] = fmaf(a[i], b.z, acc[i][2]);
                    acc[i][3] = fmaf(a[i], b.w, acc[i][3]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (mine && m0 + tr + i < Mdim && n0 + u0 + tc + j < Ndim) {
                    float* p = C + static_cast<int64_t>(m0 + tr + i) * ldc + (n0 + u0 + tc + j);
                    *p = beta ? acc[i][j] + *p : acc[i][j];
                }
        __syncwarp();
    }
}

// One k-block: six products of four steps each, the small ones first (l h', h l', m m', m h', h m', h h').
template <bool A_MN, bool B_MN, int BN>
__device__ __forceinline__ void issue_products(uint32_t d_tmem, uint32_t a0, uint32_t b0)
{
    using S = F32Shape<A_MN, B_MN, BN>;
    constexpr int A = S::TileA::kPartBytes / 16, B = S::TileB::kPartBytes / 16;       // start addresses count 16 bytes
    constexpr uint32_t idesc = umma_idesc_bf16(2 * F_BM, BN, A_MN, B_MN);
    const uint64_t da = umma_smem_desc(a0, A_MN ? F_SLAB : 16, 1024), db = umma_smem_desc(b0, B_MN ? F_SLAB : 16, 1024);
    auto product = [&](auto off_a, auto off_b, bool first) {
        constexpr int ja = A_MN ? 128 : 2, jb = B_MN ? 128 : 2, oa = decltype(off_a)::value, ob = decltype(off_b)::value;
        umma_bf16_pair_at<oa, ob>(d_tmem, da, db, idesc, !first);
        umma_bf16_pair_at<oa + ja, ob + jb>(d_tmem, da, db, idesc, true);
        umma_bf16_pair_at<oa + 2 * ja, ob + 2 * jb>(d_tmem, da, db, idesc, true);
        umma_bf16_pair_at<oa + 3 * ja, ob + 3 * jb>(d_tmem, da, db, idesc, true);
    };
    product(Int<2 * A>{}, Int<0>{}, true);
    product(Int<0>{}, Int<2 * B>{}, false);
    product(Int<A>{}, Int<B>{}, false);
    product(Int<A>{}, Int<0>{}, false);
    product(Int<0>{}, Int<B>{}, false);
    product(Int<0>{}, Int<0>{}, false);
}

template <bool A_MN, bool B_MN, int BN>
__global__ void __launch_bounds__(F_THREADS, 1)
gemm_f32_pair_kernel(const F32Operand A, const F32Operand B, float* __restrict__ C, int64_t ldc, int beta, int c_vec,
                     int Mdim, int Ndim, int Kdim, int tiles_m, int tiles_n, int* __restrict__ status)
{
    using S = F32Shape<A_MN, B_MN, BN>;
    using TileA = typename S::TileA;
    using TileB = typename S::TileB;
    constexpr int COLS = BN / 3;                             // output columns of a sum warp
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = static_cast<int>(cluster.block_rank()); // 0 = leader
    const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* tail = smem_raw + (base - raw) + F_STAGES * S::kStageBytes;
    const uint32_t full = base + F_STAGES * S::kStageBytes, done = full + 16, drained = full + 32;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tail + 48);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 56);
    uint32_t* marks = reinterpret_cast<uint32_t*>(tail + F_BARRIER_BYTES + F_SUM_WARPS * 32 * F_STAGE_PITCH * sizeof(float));

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int num_tiles = tiles_m * tiles_n;
    const int kblocks = (Kdim + F_BK - 1) / F_BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < F_STAGES; ++s) {
            mbar_init(full + 8 * s, F_OPERAND_WARPS + (rank == 0 ? 1 : 0));
            mbar_init(done + 8 * s, 1);
            mbar_init(drained + 8 * s, F_SUM_WARPS + (rank == 0 ? 1 : 0));
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    for (int i = threadIdx.x; pair + i * num_pairs < num_tiles; i += F_THREADS) marks[i] = 0;
    if (warp == F_SUM_WARPS + F_OPERAND_WARPS) {
        tmem_alloc_pair(smem_u32(tmem_slot), 2 * S::kAccCols);
        tmem_relinquish_pair();
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster.sync();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;

    bool failed = false;
    if (warp >= F_SUM_WARPS + F_OPERAND_WARPS) {
        // ------------------------------------------------ products of both CTAs
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(F_ISSUE_REGS));
        if (lane == 0 && rank == 0 && warp == F_SUM_WARPS + F_OPERAND_WARPS) {
            uint32_t it = 0;
            for (int tile = pair; tile < num_tiles && !failed; tile += num_pairs) {
                for (int kb = 0; kb < kblocks; ++kb, ++it) {
                    const uint32_t s = it & 1u, ph = (it >> 1) & 1u;
                    if (!mbar_wait(drained + 8 * s, ph ^ 1u, abort_flag) || !mbar_wait(full + 8 * s, ph, abort_flag)) { failed = true; break; }
                    mbar_try_wait_acquire_cluster(full + 8 * s, ph);   // complete: one probe acquires what the peer's warps wrote too
                    tc_fence_after_sync();
                    const uint32_t a0 = base + s * S::kStageBytes;
                    issue_products<A_MN, B_MN, BN>(tmem_base + s * S::kAccCols, a0, a0 + 3 * TileA::kPartBytes);
                    umma_commit_pair(done + 8 * s);
                }
            }
            if (failed) *abort_flag = 1;
        } else if (lane == 0 && rank == 1 && warp < F_SUM_WARPS + F_OPERAND_WARPS + 2) {
            const uint32_t mine = warp == F_SUM_WARPS + F_OPERAND_WARPS ? full : drained, theirs = map_to_cta(mine, 0);
            uint32_t it = 0;
            for (int tile = pair; tile < num_tiles && !failed; tile += num_pairs)
                for (int kb = 0; kb < kblocks; ++kb, ++it) {
                    if (!mbar_wait(mine + 8 * (it & 1u), (it >> 1) & 1u, abort_flag)) { failed = true; break; }
                    mbar_arrive_release_cluster(theirs + 8 * (it & 1u));
                }
            if (failed) *abort_flag = 1;
        }
    } else if (warp >= F_SUM_WARPS) {
        // ------------------------------------------------ operands
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(F_OPERAND_REGS));
        const int t = threadIdx.x - 32 * F_SUM_WARPS;
        TileA ta;
        TileB tb;
        auto start = [&](int tile) {
            const PairTile t0 = pair_tile(tile, tiles_m, tiles_n, 2 * F_BM, BN);
            ta.start(A, t0.m0 + rank * F_BM, Mdim, Kdim, t);
            tb.start(B, t0.n0 + rank * (BN / 2), Ndim, Kdim, t);
        };
        // A waits in registers while the stage is being read; B is fetched while A is split, into the registers that frees.
        float4 x[4];
        SplitOperandCheck seen;
        int tile = pair, kb = 0;
        if (tile < num_tiles) {
            start(tile);
#pragma unroll
            for (int i = 0; i < TileA::kPasses; ++i) x[i] = ta.load(A, i);
        }
        for (uint32_t it = 0; tile < num_tiles; ++it) {
            const uint32_t s = it & 1u, ph = (it >> 1) & 1u;
            if (!mbar_wait_warp(done + 8 * s, ph ^ 1u, abort_flag)) { failed = true; break; }
            const uint32_t a0 = base + s * S::kStageBytes;
#pragma unroll
            for (int i = 0; i < TileA::kPasses; ++i) {
                TileA::store(a0, i, t, x[i], seen);
                if (i < TileB::kPasses) x[i] = tb.load(B, i);
            }
#pragma unroll
            for (int i = 0; i < TileB::kPasses; ++i) TileB::store(a0 + 3 * TileA::kPartBytes, i, t, x[i], seen);
            if (kb + 1 == kblocks) {
                const uint32_t flags = (__any_sync(0xffffffffu, seen.flags() & SPLIT_TINY) ? SPLIT_TINY : 0u) |
                                       (__any_sync(0xffffffffu, seen.flags() & SPLIT_BIG) ? SPLIT_BIG : 0u);
                if (flags && lane == 0) flag_tile(marks + (tile - pair) / num_pairs, flags << F_FLAG_SHIFT);
                seen = SplitOperandCheck();
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(full + 8 * s);
            if (++kb < kblocks) {
                ta.advance(A);
                tb.advance(B);
            } else {
                kb = 0;
                tile += num_pairs;
                if (tile >= num_tiles) break;
                start(tile);
            }
#pragma unroll
            for (int i = 0; i < TileA::kPasses; ++i) x[i] = ta.load(A, i);
        }
        if (failed) *abort_flag = 1;
    } else {
        // ------------------------------------------------ sums
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(F_SUM_REGS));
        const int quarter = warp & 3, third = warp >> 2;
        float* stage = reinterpret_cast<float*>(tail + F_BARRIER_BYTES) + warp * 32 * F_STAGE_PITCH;
        const uint32_t taddr = tmem_base + third * COLS + (static_cast<uint32_t>(quarter * 32) << 16);
        uint32_t it = 0;
        uint32_t* mark = marks;
        for (int tile = pair; tile < num_tiles && !failed; tile += num_pairs, ++mark) {
            float sum[COLS];
#pragma unroll
            for (int c = 0; c < COLS; ++c) sum[c] = 0.f;
            for (int kb = 0; kb < kblocks; ++kb, ++it) {
                const uint32_t s = it & 1u, ph = (it >> 1) & 1u;
                if (!mbar_wait_warp(done + 8 * s, ph, abort_flag, 64)) { failed = true; break; }
                tc_fence_after_sync();
#pragma unroll
                for (int c = 0; c < COLS; c += 8) {
                    uint32_t r[8];
                    tmem_ld_32x8(taddr + s * S::kAccCols + c, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 8; ++e) sum[c + e] += __uint_as_float(r[e]);
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(drained + 8 * s);
            }
            if (failed) break;
            const PairTile t0 = pair_tile(tile, tiles_m, tiles_n, 2 * F_BM, BN);
            const int m0 = t0.m0 + rank * F_BM + quarter * 32, n0 = t0.n0 + third * COLS;
            const uint32_t operands = *const_cast<volatile uint32_t*>(mark) >> F_FLAG_SHIFT;
            SplitOutputCheck check;
#pragma unroll
            for (int c = 0; c < COLS; ++c) check.add(sum[c]);
            // Columns beyond the matrix are not finite where their row has others that are not, or zeros: looked at again for nothing at worst.
            if (__any_sync(0xffffffffu, m0 + lane < Mdim && n0 < Ndim && check.suspect(operands, Kdim))) {
                if (lane == 0) atomicOr(mark, 1u << warp);
                continue;
            }
            float* crow = C + static_cast<int64_t>(m0 + lane) * ldc + n0;
#pragma unroll
            for (int c = 0; c < COLS; c += 16) {
                const int valid = Ndim - (n0 + c);
                if (m0 >= Mdim || valid <= 0) continue;      // the same for the whole warp
                if (!c_vec) {
#pragma unroll
                    for (int e = 0; e < 16; ++e) stage[lane * F_STAGE_PITCH + e] = sum[c + e];
                    __syncwarp();
                    // A row at a time, half a warp each: consecutive lanes to consecutive columns.
                    const int e = lane & 15;
                    if (e < valid) {
                        float* p = C + static_cast<int64_t>(m0 + (lane >> 4)) * ldc + n0 + c + e;
                        for (int i = lane >> 4; i < 32 && m0 + i < Mdim; i += 2, p += 2 * ldc) {
                            const float f = stage[i * F_STAGE_PITCH + e];
                            *p = beta ? f + *p : f;
                        }
                    }
                    __syncwarp();
                } else if (m0 + lane < Mdim) {
                    float* p = crow + c;
                    if (valid >= 16) {
#pragma unroll
                        for (int h = 0; h < 16; h += 8) {
                            float y[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) y[e] = sum[c + h + e];
                            if (beta) {
                                const float4 u = *reinterpret_cast<const float4*>(p + h), w = *reinterpret_cast<const float4*>(p + h + 4);
                                y[0] += u.x; y[1] += u.y; y[2] += u.z; y[3] += u.w;
                                y[4] += w.x; y[5] += w.y; y[6] += w.z; y[7] += w.w;
                            }
                            store_f32x8(p + h, y);
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            if (e < valid) p[e] = beta ? sum[c + e] + p[e] : sum[c + e];
                    }
                }
            }
        }
        if (failed) *abort_flag = 1;
        // Marked outputs: every product is done, the ring is free, and nobody waits but for the end.  All sum warps get here.
        __syncwarp();
        if (!sum_warps_any(failed)) {
            mark = marks;
            for (int tile = pair; tile < num_tiles; tile += num_pairs, ++mark) {
                if (!(*mark & ((1u << F_SUM_WARPS) - 1u))) continue;
                const PairTile t0 = pair_tile(tile, tiles_m, tiles_n, 2 * F_BM, BN);
                redo_tile<A_MN, B_MN, BN>(A, B, C, ldc, beta, t0.m0 + rank * F_BM, t0.n0, Mdim, Ndim, Kdim, *mark,
                                          reinterpret_cast<float*>(smem_raw + (base - raw)));
            }
        }
    }
    if (failed && status) atomicExch(status, VELORA_ERR_TIMEOUT);

    tc_fence_before_sync();
    __syncthreads();
    cluster.sync();                                          // nobody signals or reads a CTA that has left
    tc_fence_after_sync();
    if (warp == F_SUM_WARPS + F_OPERAND_WARPS) {
        __syncwarp();
        tmem_dealloc_pair(tmem_base, 2 * S::kAccCols);
    }
}

template <bool A_MN, bool B_MN, int BN>
int launch_shape(const F32Operand& A, const F32Operand& B, float* C, int64_t ldc, int beta, int Mdim, int Ndim, int Kdim,
                 int* status, const DeviceInfo& di, cudaStream_t stream)
{
    constexpr size_t smem = F32Shape<A_MN, B_MN, BN>::kSmem;
    if (static_cast<size_t>(di.smem_optin) < smem || di.sm_count < 2) return VELORA_ERR_UNSUPPORTED;
    static DeviceOnce configured;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return VELORA_ERR_CUDA;
    auto kern = gemm_f32_pair_kernel<A_MN, B_MN, BN>;
    if (!configured.get(dev)) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess) return VELORA_ERR_CUDA;
        configured.set(dev);
    }
    const int tiles_m = static_cast<int>(ceil_div64(Mdim, 2 * F_BM)), tiles_n = static_cast<int>(ceil_div64(Ndim, BN));
    const int64_t tiles = static_cast<int64_t>(tiles_m) * tiles_n;
    const int pairs = tiles < di.sm_count / 2 ? static_cast<int>(tiles) : di.sm_count / 2;
    if (ceil_div64(tiles, pairs) > F32Shape<A_MN, B_MN, BN>::kMaxTiles) {             // 7 GB of outputs and more: half of the rows at a time
        if (tiles_m < 2) return VELORA_ERR_UNSUPPORTED;
        const int rows = tiles_m / 2 * 2 * F_BM;
        const F32Operand A2{A.p + static_cast<int64_t>(rows) * (A_MN ? 1 : A.ld), A.ld, A.vec};
        const int rc = launch_shape<A_MN, B_MN, BN>(A, B, C, ldc, beta, rows, Ndim, Kdim, status, di, stream);
        return rc != VELORA_OK ? rc : launch_shape<A_MN, B_MN, BN>(A2, B, C + rows * ldc, ldc, beta, Mdim - rows, Ndim, Kdim, status, di, stream);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(2 * pairs), 1, 1);
    cfg.blockDim = dim3(F_THREADS, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int c_vec = c_rows_vec(C, ldc, sizeof(float)) ? 1 : 0;
    if (cudaLaunchKernelEx(&cfg, kern, A, B, C, ldc, beta, c_vec, Mdim, Ndim, Kdim, tiles_m, tiles_n, status) != cudaSuccess) {
        cudaGetLastError();
        return VELORA_ERR_UNSUPPORTED;                       // a refused cluster: the CUDA cores
    }
    return after_launch();
}

}  // namespace

int launch_gemm_f32_tc(int kind, const void* A, int64_t lda, const void* B, int64_t ldb, void* C, int64_t ldc, int beta,
                       int64_t Mdim, int64_t Ndim, int64_t Kdim, int* status, cudaStream_t stream)
{
    if (Mdim < 1 || Ndim < 1 || Kdim < 1) return VELORA_ERR_UNSUPPORTED;
    // Indexes of a tile's far edge stay within 32 bits, and so do the tiles.
    if (Mdim > (1 << 30) || Ndim > (1 << 30) || Kdim > (1 << 30)) return VELORA_ERR_UNSUPPORTED;
    if (ceil_div64(Mdim, 2 * F_BM) * ceil_div64(Ndim, 96) > (1 << 30)) return VELORA_ERR_UNSUPPORTED;
    DeviceInfo di;
    const int rc = device_info(&di);
    if (rc != VELORA_OK) return rc;
    const F32Operand a{static_cast<const float*>(A), lda, aligned16(A) && lda % 4 == 0 ? 1 : 0};
    const F32Operand b{static_cast<const float*>(B), ldb, aligned16(B) && ldb % 4 == 0 ? 1 : 0};
    const int m = static_cast<int>(Mdim), n = static_cast<int>(Ndim), k = static_cast<int>(Kdim);
    float* c = static_cast<float*>(C);
    // By estimated time in microseconds, from what both forms take between 256 x 64, K = 64 and 12608 x 768, K = 768.  A k-block costs
    // nearly the same at both widths (24 products of no less than 97 cycles each), so tiles of 96 columns pay only where those of 192
    // leave pairs idle.  Measured, us, 192 / 96 / CUDA cores: 12608 x 768, K = 768: 97 / 142 / 373; 2048 x 768, K = 768: 39 / 34 / 94;
    // 3000 x 3000, K = 100: 31 / 40 / 55; 1280 x 440, K = 300: 21 / 19 / 19; 640 x 256, K = 256: 21 / 17 / 13.
    const int64_t kblocks = ceil_div64(Kdim, F_BK), tiles_m = ceil_div64(Mdim, 2 * F_BM), pairs = di.sm_count / 2 > 0 ? di.sm_count / 2 : 1;
    const double us192 = 6.0 + ceil_div64(tiles_m * ceil_div64(Ndim, 192), pairs) * (2.2 * kblocks + 4.5);
    const double us96 = 6.5 + ceil_div64(tiles_m * ceil_div64(Ndim, 96), pairs) * (1.95 * kblocks + 1.5);
    const int bn = us96 < us192 ? 96 : 192;
    if (0.95 * gemm_simt_f32_us(Mdim, Ndim, Kdim, di.sm_count) < (bn == 96 ? us96 : us192)) return VELORA_ERR_UNSUPPORTED;
#define VELORA_F32_CASE(AMN, BMN)                                                                             \
    return bn == 192 ? launch_shape<AMN, BMN, 192>(a, b, c, ldc, beta, m, n, k, status, di, stream)           \
                     : launch_shape<AMN, BMN, 96>(a, b, c, ldc, beta, m, n, k, status, di, stream)
    if (kind == GEMM_NT_K_K) { VELORA_F32_CASE(false, false); }
    if (kind == GEMM_NN_K_MN) { VELORA_F32_CASE(false, true); }
    VELORA_F32_CASE(true, true);
#undef VELORA_F32_CASE
}

}  // namespace velora
