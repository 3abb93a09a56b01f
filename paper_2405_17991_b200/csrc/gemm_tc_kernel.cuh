// The single-CTA tensor-core product (sm_100a): C[Mdim, Ndim] = A * B with bf16 operands and fp32 accumulation.
//
// One persistent, warp-specialised kernel, output tile 128 x BN, K step 64.  Warp 0 feeds a shared-memory ring with TMA
// tile loads (128-byte swizzle); warp 1 issues tcgen05.mma (M = 128, N = BN, K = 16) into one of two TMEM
// accumulators; warps 2..5 drain the other one with tcgen05.ld, convert and store, so the epilogue of a tile overlaps
// the main loop of the next.  Either operand may be K-major (rows contiguous along K) or MN-major (rows contiguous
// along M or N): the latter is loaded as 64 x 64 boxes and consumed through an MN-major matrix descriptor, so no
// transpose pass exists.  Ragged edges rely on TMA zero fill for loads and on predicated stores.
//
// Outputs of few tiles: narrower tiles (BN = 64, 128, 192) and up to eight CTAs of a cluster per tile, each with its share
// of the contraction.  Each parks its partial tile in its own shared memory (the ring is idle by then) and, behind a
// cluster barrier, adds all of them up for its share of the rows, in a fixed order.  A 386 x 320 output with K = 9032
// was 8 CTAs of 142 k-blocks (53 us).
#pragma once

#include <cooperative_groups.h>

#include "gemm_fuse.cuh"
#include "gemm_store.cuh"
#include "gemm_tc.cuh"
#include "tc_common.cuh"

namespace velora {

using namespace tc;

namespace {

constexpr int BM = 128, BK = 64;
constexpr int A_BYTES = BM * BK * 2;              // 16 KB
constexpr int SLAB_BYTES = 64 * BK * 2;           // one 64-wide MN-major slab: 64 k-rows x 128 bytes
constexpr int MAX_SPLITS = 8;                     // the portable cluster size
constexpr int GEMM_THREADS = 192;                   // producer, issuer, four epilogue warps
constexpr int GEMM_THREADS_SHORT = 320;             // eight epilogue warps, for contractions of up to SHORT_KBLOCKS k-blocks
constexpr int SHORT_KBLOCKS = 8;
constexpr int FUSE_THREADS = 384;    // + four compress warps (6, 7, 10, 11) and two idle ones (8, 9)
constexpr int BARRIER_BYTES = 256;

// What depends on the tile's width: as many stages as fit 200 KB, at most eight.
template <int BN> struct TileShape {
    static constexpr int kBBytes = BN * BK * 2;
    static constexpr int kFit = 200 * 1024 / (A_BYTES + kBBytes);
    static constexpr int kStages = kFit < 8 ? kFit : 8;
    static constexpr int kTmemCols = BN > 128 ? 512 : (BN > 64 ? 256 : 128);       // two accumulators, a power of two
    // Behind the ring: output blocks on their way to memory, of eight warps (four at BN = 192, whose ring has the room of the
    // others) or, unaligned rows, of four.
    static constexpr int kStoreWarps = BN == 192 ? 4 : 8;
    static constexpr int kStagingBytes = kStoreWarps == 8 ? 8 * kStoreBytes : 17 * 1024;
    static_assert(kStagingBytes >= 4 * kStageFloats * 4 && kStagingBytes >= kStoreWarps * kStoreBytes && kStagingBytes % 1024 == 0, "staging");
    static constexpr size_t kSmem = 1024 + static_cast<size_t>(kStages) * (A_BYTES + kBBytes) + kStagingBytes + BARRIER_BYTES;
    static constexpr int kPartialPitch = BN + 4;                                    // floats per row of a parked partial tile
    static_assert(static_cast<size_t>(BM) * kPartialPitch * 4 <= static_cast<size_t>(kStages) * (A_BYTES + kBBytes), "fits the ring");
};

struct TileCoord {
    int m0, n0;
};

// Tiles are walked in bands of 8 m-tiles so that CTAs running together share B tiles in L2.
template <int BN>
__device__ __forceinline__ TileCoord tile_coord(int tile, int tiles_m, int tiles_n)
{
    constexpr int BAND = 8;
    const int per_band = BAND * tiles_n;
    const int band = tile / per_band;
    const int in_band = tile - band * per_band;
    const int band_rows = (tiles_m - band * BAND < BAND) ? tiles_m - band * BAND : BAND;
    const int tn = in_band / band_rows;
    const int tm = band * BAND + (in_band - tn * band_rows);
    return {tm * BM, tn * BN};
}

// FUSE = 0: plain GEMM.  FUSE = 1 / 2 / 3 (forward only, A = X K-major): Z = compress(X, v) (fp32 / bf16 /
// E4M3 storage) is computed by four extra warps for the row block the CTA is multiplying, from lines of X
// that are on their way through L2 for the GEMM anyway, so X crosses HBM once for both results.  The CTA
// working on n-tile j handles the sub-token groups g with g % tiles_n == j, so the work is spread over the
// CTAs that share a row block.  The compress warps read X with plain 16-byte loads and keep v in registers:
// they share no stage and no barrier with the GEMM's pipeline, only the pipe of their shuffles (gemm_fuse.cuh),
// and they sit on warps 6, 7, 10, 11 so that none of them shares a warp scheduler (warp % 4) with the TMA
// producer (warp 0) or the MMA issuer (warp 1).
template <bool A_MN, bool B_MN, typename CT, int FUSE, int BN>
__global__ void __launch_bounds__(FUSE ? FUSE_THREADS : GEMM_THREADS_SHORT, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmC, CT* __restrict__ C, int64_t ldc, int beta, int Mdim, int Ndim, int Kdim,
               int tiles_m, int tiles_n, int kb_per_split, int c_vec, int* __restrict__ status, const FuseArgs fz)
{
    typedef TileShape<BN> S;
    constexpr int B_BYTES = S::kBBytes, STAGES = S::kStages, TMEM_COLS = S::kTmemCols;
    static_assert(FUSE == 0 || (!A_MN && !B_MN), "compress rides on the K-major forward GEMM only");
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;               // swizzled tiles need 1024-byte alignment
    uint8_t* smem = smem_raw + (base - raw);
    const uint32_t sA = base;
    const uint32_t sB = base + STAGES * A_BYTES;
    uint8_t* staging = smem + STAGES * (A_BYTES + B_BYTES);
    uint8_t* tail = staging + S::kStagingBytes;
    const uint32_t bars = base + STAGES * (A_BYTES + B_BYTES) + S::kStagingBytes;
    const uint32_t full = bars, empty = bars + 8 * STAGES;
    const uint32_t tfull = bars + 16 * STAGES, tempty = tfull + 16;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tail + 16 * STAGES + 48);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 16 * STAGES + 56);
    volatile int* tiles_started = reinterpret_cast<volatile int*>(tail + 16 * STAGES + 60);   // producer's progress, read by the compress warps

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int num_tiles = tiles_m * tiles_n;
    const int kblocks = (Kdim + BK - 1) / BK;
    const int splits = static_cast<int>(gridDim.y), split = static_cast<int>(blockIdx.y);    // split = rank in the cluster
    const int kb0 = split * kb_per_split;
    const int kb1 = kb0 + kb_per_split < kblocks ? kb0 + kb_per_split : kblocks;              // > kb0 (host)

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full + 8 * s, 1);
            mbar_init(empty + 8 * s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(tfull + 8 * a, 1);
            mbar_init(tempty + 8 * a, FUSE ? 4 : (blockDim.x - 64) / 32);        // the epilogue's warps
        }
        *abort_flag = 0;
        *tiles_started = 0;
        fence_mbar_init();
        prefetch_tensormap(&tmA);
        prefetch_tensormap(&tmB);
        if (c_vec == C_TILES) prefetch_tensormap(&tmC);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    pdl_wait();                                              // nothing in global memory has been touched so far
    if (splits == 1) pdl_trigger();

    bool failed = false;
    if (warp == 0) {
        // ------------------------------------------------ TMA producer (one lane)
        if (lane == 0) {
            uint32_t it = 0;
            int started = 0;
            for (int tile = blockIdx.x; tile < num_tiles && !failed; tile += gridDim.x) {
                if (FUSE) *tiles_started = ++started;          // the compress warps may take this tile's row block now
                const TileCoord tc0 = tile_coord<BN>(tile, tiles_m, tiles_n);
                for (int kb = kb0; kb < kb1; ++kb, ++it) {
                    const uint32_t s = it % STAGES, ph = (it / STAGES) & 1u;
                    if (!mbar_wait(empty + 8 * s, ph ^ 1u, abort_flag)) { failed = true; break; }
                    mbar_arrive_expect_tx(full + 8 * s, A_BYTES + B_BYTES);
                    const int k0 = kb * BK;
                    if (A_MN) {
#pragma unroll
                        for (int i = 0; i < BM / 64; ++i)
                            tma_load_2d(sA + s * A_BYTES + i * SLAB_BYTES, &tmA, full + 8 * s, tc0.m0 + 64 * i, k0);
                    } else {
                        tma_load_2d(sA + s * A_BYTES, &tmA, full + 8 * s, k0, tc0.m0);
                    }
                    if (B_MN) {
#pragma unroll
                        for (int i = 0; i < BN / 64; ++i)
                            tma_load_2d(sB + s * B_BYTES + i * SLAB_BYTES, &tmB, full + 8 * s, tc0.n0 + 64 * i, k0);
                    } else {
                        tma_load_2d(sB + s * B_BYTES, &tmB, full + 8 * s, k0, tc0.n0);
                    }
                }
            }
            if (failed) {
                *abort_flag = 1;
                // Let this CTA's own copies in flight land before shared memory is given up.
                const uint32_t back = it < STAGES ? it : STAGES;
                for (uint32_t j = 1; j <= back; ++j) {
                    const uint32_t jt = it - j;
                    const unsigned long long t0 = globaltimer_ns();
                    while (!mbar_try_wait(full + 8 * (jt % STAGES), (jt / STAGES) & 1u))
                        if (globaltimer_ns() - t0 > kWaitLimitNs) break;
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer (one lane)
        if (lane == 0) {
            constexpr uint32_t idesc = umma_idesc_bf16(BM, BN, A_MN, B_MN);
            uint32_t it = 0, t = 0;
            for (int tile = blockIdx.x; tile < num_tiles && !failed; tile += gridDim.x, ++t) {
                const uint32_t acc = t & 1u, aph = (t >> 1) & 1u;
                if (!mbar_wait(tempty + 8 * acc, aph ^ 1u, abort_flag)) { failed = true; break; }
                tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + acc * BN;
                for (int kb = kb0; kb < kb1; ++kb, ++it) {
                    const uint32_t s = it % STAGES, ph = (it / STAGES) & 1u;
                    if (!mbar_wait(full + 8 * s, ph, abort_flag)) { failed = true; break; }
                    tc_fence_after_sync();
                    const uint32_t a_addr = sA + s * A_BYTES, b_addr = sB + s * B_BYTES;
#pragma unroll
                    for (int j = 0; j < BK / 16; ++j) {
                        // K-major: 16 elements of K = 32 bytes inside the swizzled 128-byte row.
                        // MN-major: 16 k-rows of 128 bytes; 64-wide slabs are BK*128 bytes apart.
                        const uint64_t da = A_MN ? umma_smem_desc(a_addr + j * 2048, SLAB_BYTES, 1024)
                                                 : umma_smem_desc(a_addr + j * 32, 16, 1024);
                        const uint64_t db = B_MN ? umma_smem_desc(b_addr + j * 2048, SLAB_BYTES, 1024)
                                                 : umma_smem_desc(b_addr + j * 32, 16, 1024);
                        umma_bf16(d_tmem, da, db, idesc, kb != kb0 || j != 0);
                    }
                    umma_commit(empty + 8 * s);           // the stage is free once these MMAs have read it
                }
                if (failed) break;
                umma_commit(tfull + 8 * acc);             // the accumulator is complete
            }
            if (failed) *abort_flag = 1;
        }
    } else if (FUSE && (warp == 8 || warp == 9)) {
        // Idle on purpose: these two would share warp schedulers 0 and 1 with the producer and the MMA issuer.
    } else if (FUSE && warp >= 6) {
        // ------------------------------------------------ compress (4 warps, 32 rows of the tile's 128 each)
        const int cwi = warp < 8 ? warp - 6 : warp - 8;
        const int cpr = (fz.Dsub >> 3) < 8 ? 8 : (fz.Dsub >> 3);
        const int n_groups = (Kdim + 8 * cpr - 1) / (8 * cpr);
        auto walk = [&](auto vs) {
            vs.load(fz.v, fz.Dsub, lane);
            int ti = 0;
            for (int tile = blockIdx.x; tile < num_tiles; tile += gridDim.x, ++ti) {
                if (!wait_for_tile(tiles_started, ti, abort_flag)) { failed = true; break; }
                const TileCoord tc0 = tile_coord<BN>(tile, tiles_m, tiles_n);
                const int r0 = tc0.m0 + cwi * 32;
                CompressWalk<FUSE, vs.kParts>(fz, vs, r0, Mdim, Kdim, lane).run(tc0.n0 / BN * splits + split, tiles_n * splits, n_groups);
            }
        };
        if (fz.Dsub <= 256) walk(VSlice<1>{});
        else if (fz.Dsub == 512) walk(VSlice<2>{});
        else walk(VSlice<4>{});
    } else {
        // ------------------------------------------------ epilogue (one TMEM lane quarter per warp; short contractions have
        // two sets of four warps, which take the 64-column steps in turn: 22 -> 20 us for 8192 x 4096 with K = 16, no gain at
        // K = 3072)
        const int quarter = warp & 3;
        const int set = FUSE ? 0 : (warp - 2) >> 2;
        const int sets = FUSE || blockDim.x == GEMM_THREADS || (sizeof(CT) == 2 && !c_vec && splits == 1) ? 1 : 2;     // staging room for four warps
        const uint32_t block = smem_u32(staging) + (warp - 2) * kStoreBytes;
        uint32_t t = 0;
        for (int tile = blockIdx.x; tile < num_tiles && !failed; tile += gridDim.x, ++t) {
            const TileCoord tc0 = tile_coord<BN>(tile, tiles_m, tiles_n);
            const uint32_t acc = t & 1u, aph = (t >> 1) & 1u;
            if (!mbar_wait_warp(tfull + 8 * acc, aph, abort_flag, 256)) { failed = true; break; }
            tc_fence_after_sync();
            const int row = tc0.m0 + quarter * 32 + lane;
            const uint32_t taddr = tmem_base + acc * BN + (static_cast<uint32_t>(quarter * 32) << 16);
            if (splits > 1) {                                 // one tile per CTA: park the partial product
                float* prow = reinterpret_cast<float*>(smem) + (quarter * 32 + lane) * S::kPartialPitch;
#pragma unroll 1
                for (int c = set; c < BN / 32; c += sets) {
                    uint32_t r[32];
                    tmem_ld_32x32(taddr + c * 32, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        *reinterpret_cast<uint4*>(prow + c * 32 + 4 * i) = make_uint4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
                }
                continue;
            }
            CT* crow = C + static_cast<int64_t>(row) * ldc + tc0.n0;
            const int last = set >= sets ? -1 : ((BN / 64 - 1 - set) / sets * sets + set) * 2;    // this warp's last step
            if (last < 0 || set >= BN / 64) {                 // nothing for this set in a tile of this width
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty + 8 * acc);
                continue;
            }
#pragma unroll 1
            for (int c = 2 * set; c < BN / 32; c += 2 * sets) {       // 64 columns a step: two TMEM loads in flight
                uint32_t r[2][32];
                tmem_ld_32x32(taddr + c * 32, r[0]);
                tmem_ld_32x32(taddr + c * 32 + 32, r[1]);
                tmem_ld_wait();
                if (c == last) {                              // this warp has read its share: hand it back
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty + 8 * acc);
                }
                const int valid = Ndim - (tc0.n0 + c * 32);
                if (sizeof(CT) == 2 && c_vec == C_TILES && (valid >= 64 || Ndim % 8 == 0)) {
                    if (row - lane < Mdim && valid > 0) store_block(&tmC, block, r, tc0.n0 + c * 32, row - lane, lane);
                } else if (sizeof(CT) == 4 || c_vec) {            // fp32 rows always are (host)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        if (row < Mdim && valid > 32 * h) Store32<CT>::run(crow + (c + h) * 32, r[h], valid - 32 * h, beta);
                } else if (row - lane < Mdim) {
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        if (valid > 32 * h)
                            store_rows_staged<CT>(crow - static_cast<int64_t>(lane) * ldc + (c + h) * 32, ldc, Mdim - (row - lane), valid - 32 * h,
                                                  r[h], beta, reinterpret_cast<float*>(staging) + quarter * kStageFloats, lane);
                }
            }
        }
        if (sizeof(CT) == 2 && c_vec == C_TILES && lane == 0) bulk_wait_all();
        if (failed) *abort_flag = 1;
    }
    if (failed && status) atomicExch(status, VELORA_ERR_TIMEOUT);

    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == 1) {
        __syncwarp();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
    if (splits > 1) {
        // Every CTA reaches both cluster barriers whatever happened above.
        namespace cg = cooperative_groups;
        cg::cluster_group cluster = cg::this_cluster();
        cluster.sync();                                      // all partials of the tile are in shared memory
        const TileCoord tc0 = tile_coord<BN>(blockIdx.x, tiles_m, tiles_n);
        const int rows_per = (BM + splits - 1) / splits;
        const int r_begin = split * rows_per;
        int r_end = r_begin + rows_per < BM ? r_begin + rows_per : BM;
        if (r_end > Mdim - tc0.m0) r_end = Mdim - tc0.m0;
        const float* part = reinterpret_cast<const float*>(smem);
        for (int idx = threadIdx.x; idx < (r_end - r_begin) * (BN / 4); idx += blockDim.x) {
            const int r = r_begin + idx / (BN / 4), col = idx % (BN / 4) * 4;
            const int left = Ndim - (tc0.n0 + col);
            if (left <= 0) continue;
            float4 x[MAX_SPLITS];
#pragma unroll
            for (int s = 0; s < MAX_SPLITS; ++s)
                if (s < splits) x[s] = *reinterpret_cast<const float4*>(cluster.map_shared_rank(part, s) + r * S::kPartialPitch + col);
            float y[4] = {x[0].x, x[0].y, x[0].z, x[0].w};
#pragma unroll
            for (int s = 1; s < MAX_SPLITS; ++s)               // fixed order
                if (s < splits) { y[0] += x[s].x; y[1] += x[s].y; y[2] += x[s].z; y[3] += x[s].w; }
            CT* p = C + static_cast<int64_t>(tc0.m0 + r) * ldc + tc0.n0 + col;
            if (c_vec && left >= 4) {
                Store4<CT>::run(p, y, beta);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (e < left) {
                        float f = y[e];
                        if (beta) f += Elem<CT>::load(p + e);
                        Elem<CT>::store(p + e, f);
                    }
            }
        }
        cluster.sync();                                      // nobody leaves while its partial is still being read
    }
}

template <bool A_MN, bool B_MN, typename CT, int FUSE, int BN>
int launch_kernel(const CUtensorMap& ta, const CUtensorMap& tb, void* C, int64_t ldc, int beta,
                  int Mdim, int Ndim, int Kdim, int splits, int* status, cudaStream_t stream, const FuseArgs fz = FuseArgs{})
{
    typedef TileShape<BN> S;
    static DeviceOnce configured;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return VELORA_ERR_CUDA;
    auto kern = gemm_tc_kernel<A_MN, B_MN, CT, FUSE, BN>;
    if (!configured.get(dev)) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(S::kSmem)) != cudaSuccess)
            return VELORA_ERR_CUDA;
        configured.set(dev);
    }
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc != VELORA_OK) return rc;
    const int tiles_m = (Mdim + BM - 1) / BM, tiles_n = (Ndim + BN - 1) / BN;
    const int64_t tiles = static_cast<int64_t>(tiles_m) * tiles_n;
    const int kblocks = (Kdim + BK - 1) / BK;
    const int threads = FUSE ? FUSE_THREADS : (kblocks <= SHORT_KBLOCKS * splits ? GEMM_THREADS_SHORT : GEMM_THREADS);
    int c_vec = c_rows_vec(C, ldc, sizeof(CT)) ? C_VECTORS : C_ELEMENTS;
    // bf16 rows on 16-byte boundaries leave as tiles.
    CUtensorMap tc = ta;
    if (sizeof(CT) == 2 && c_vec && !beta && splits <= 1 && ((threads - 64) / 32 <= S::kStoreWarps || FUSE) && tc_operand_ok(C, ldc) &&
        make_tmap_bf16_2d(&tc, C, Ndim, Mdim, ldc, 64, 32) == VELORA_OK)
        c_vec = C_TILES;
    if (splits <= 1) {
        const int grid = static_cast<int>(tiles < di.sm_count ? tiles : di.sm_count);
        return launch_chained(kern, dim3(static_cast<unsigned>(grid)), threads, S::kSmem, stream,
                              ta, tb, tc, static_cast<CT*>(C), ldc, beta, Mdim, Ndim, Kdim, tiles_m, tiles_n, kblocks, c_vec, status, fz);
    }
    const int kb_per_split = (kblocks + splits - 1) / splits;
    splits = (kblocks + kb_per_split - 1) / kb_per_split;             // no split without k-blocks
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(tiles), static_cast<unsigned>(splits), 1);
    cfg.blockDim = dim3(static_cast<unsigned>(threads), 1, 1);
    cfg.dynamicSmemBytes = S::kSmem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = static_cast<unsigned>(splits);
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, ta, tb, tc, static_cast<CT*>(C), ldc, beta, Mdim, Ndim, Kdim, tiles_m, tiles_n, kb_per_split, c_vec,
                           status, fz) != cudaSuccess) {
        cudaGetLastError();                                           // a refused cluster: the same tiles, one CTA each
        return launch_kernel<A_MN, B_MN, CT, FUSE, BN>(ta, tb, C, ldc, beta, Mdim, Ndim, Kdim, 1, status, stream, fz);
    }
    return after_launch();
}

}  // namespace
}  // namespace velora
