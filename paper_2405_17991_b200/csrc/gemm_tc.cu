// Dense products of Algorithm 1 (arxiv 2405.17991) on the sm_100a tensor cores, host side:
//   Y = X W^T (forward), dX = dY W (input gradient), dW = dY^T Xhat (explicit weight gradient).
// The choice between the CTA-pair kernel (gemm_tc2.cu) and the single-CTA kernel's shapes
// (gemm_tc_kernel.cuh), and the routes of the forward.
#include "gemm_tc_kernel.cuh"

namespace velora {

// The shape a product runs in, by estimated time in microseconds: waves of tiles, each the CTA's k-blocks (0.39 a k-block
// of a 256 x 256 pair tile and 0.43 of 128 x 256 on large products; narrower tiles are held back by their operand loads)
// and half a microsecond between tiles, plus the last tile's epilogue, the cluster launch of a pair, and for a split
// contraction the exchange of the partial tiles.  Splits only where every cluster of the grid is resident at once:
// clusters do not straddle the groups of 16 or more SMs.
// Measured, us, against the pair kernel (128 x 256 tiles below 74 pair tiles): 615 x 296, K = 4536: 46 -> 13; 2114 x 576,
// K = 4096: 26 -> 23; 12608 x 768, K = 3072 (150 pair tiles on 74 pairs, now 396 tiles of 192): 56 -> 53.
GemmShape gemm_shape(int64_t Mdim, int64_t Ndim, int64_t Kdim, int sm_count, bool fused)
{
    static const struct { int bn; double per_kblock; } kSingle[] = {{256, 0.43}, {192, 0.34}, {128, 0.28}, {64, 0.19}};
    const int64_t kblocks = ceil_div64(Kdim, BK), tiles_m = ceil_div64(Mdim, BM);
    GemmShape best{true, 256, 1};
    double best_us = static_cast<double>(ceil_div64(ceil_div64(Mdim, 256) * ceil_div64(Ndim, 256), sm_count / 2)) * (kblocks * 0.39 + 0.5) + 3.5;
    for (const auto& c : kSingle) {
        if (fused && c.bn != 256 && c.bn != 128) continue;
        const int64_t tiles = tiles_m * ceil_div64(Ndim, c.bn);
        if (tiles > (1 << 30)) continue;
        for (int s = 1; s <= MAX_SPLITS && s <= kblocks; ++s) {
            if (s > 1 && tiles > static_cast<int64_t>(sm_count / 18) * (16 / s)) break;
            const double us = static_cast<double>(ceil_div64(tiles, sm_count)) * (ceil_div64(kblocks, s) * c.per_kblock + 0.5) +
                              2.0 * c.bn / 256 + (s > 1 ? 2.5 + 1.5 * c.bn / 256 : 0.0);
            if (us < best_us - 0.2) {
                best_us = us;
                best = GemmShape{false, c.bn, s};
            }
        }
    }
    return best;
}

bool tc_operand_ok(const void* p, int64_t ld_elems)
{
    return aligned16(p) && ld_elems % 8 == 0 && ld_elems * 2 < (static_cast<int64_t>(1) << 40);
}

int launch_gemm_tc(int kind, const void* A, int64_t lda, const void* B, int64_t ldb,
                   void* C, int c_dtype, int64_t ldc, int beta,
                   int64_t Mdim, int64_t Ndim, int64_t Kdim, int in_dtype, int* status, cudaStream_t stream)
{
    if (in_dtype == VELORA_F32 && c_dtype == VELORA_F32)
        return launch_gemm_f32_tc(kind, A, lda, B, ldb, C, ldc, beta, Mdim, Ndim, Kdim, status, stream);
    if (in_dtype != VELORA_BF16) return VELORA_ERR_UNSUPPORTED;
    if (Mdim < 1 || Ndim < 1 || Kdim < 1) return VELORA_ERR_UNSUPPORTED;
    if (Mdim > (1 << 30) || Ndim > (1 << 30) || Kdim > (1 << 30)) return VELORA_ERR_UNSUPPORTED;
    if (!tc_operand_ok(A, lda) || !tc_operand_ok(B, ldb)) return VELORA_ERR_UNSUPPORTED;
    // An fp32 result on rows that vector stores cannot write stays with the CUDA-core product, whose sums are rounded and
    // not truncated (relative error of 8192 positive terms: 1.6e-7, 3.5e-5 here); a bf16 result hides the difference.
    if (c_dtype == VELORA_F32 && !c_rows_vec(C, ldc, sizeof(float))) return VELORA_ERR_UNSUPPORTED;
    if ((static_cast<int64_t>((Mdim + BM - 1) / BM) * ((Ndim + 255) / 256)) > (1 << 30)) return VELORA_ERR_UNSUPPORTED;

    DeviceInfo di;
    int rc = device_info(&di);
    if (rc != VELORA_OK) return rc;
    GemmShape shape = gemm_shape(Mdim, Ndim, Kdim, di.sm_count, false);
    if (shape.pair) {
        const int prc = launch_gemm_tc_pair(kind, A, lda, B, ldb, C, c_dtype, ldc, beta, Mdim, Ndim, Kdim, in_dtype, status, stream);
        if (prc != VELORA_ERR_UNSUPPORTED) return prc;
        shape = GemmShape{false, 256, 1};
    }
    const bool a_mn = (kind == GEMM_TN_MN_MN);
    const bool b_mn = (kind != GEMM_NT_K_K);
    CUtensorMap ta, tb;
    // K-major operand: [rows = M or N][K], box 64 (K) x tile rows.  MN-major: [K][M or N], box 64 x 64.
    rc = a_mn ? make_tmap_bf16_2d(&ta, A, Mdim, Kdim, lda, 64, BK) : make_tmap_bf16_2d(&ta, A, Kdim, Mdim, lda, BK, BM);
    if (rc != VELORA_OK) return rc;
    rc = b_mn ? make_tmap_bf16_2d(&tb, B, Ndim, Kdim, ldb, 64, BK) : make_tmap_bf16_2d(&tb, B, Kdim, Ndim, ldb, BK, shape.bn);
    if (rc != VELORA_OK) return rc;

    const int m = static_cast<int>(Mdim), n = static_cast<int>(Ndim), k = static_cast<int>(Kdim);
#define VELORA_GEMM_WIDTH(AMN, BMN, CT)                                                                                          \
    switch (shape.bn) {                                                                                                          \
        case 64: return launch_kernel<AMN, BMN, CT, 0, 64>(ta, tb, C, ldc, beta, m, n, k, shape.splits, status, stream);         \
        case 128: return launch_kernel<AMN, BMN, CT, 0, 128>(ta, tb, C, ldc, beta, m, n, k, shape.splits, status, stream);       \
        case 192: return launch_kernel<AMN, BMN, CT, 0, 192>(ta, tb, C, ldc, beta, m, n, k, shape.splits, status, stream);       \
        default: return launch_kernel<AMN, BMN, CT, 0, 256>(ta, tb, C, ldc, beta, m, n, k, shape.splits, status, stream);        \
    }
#define VELORA_GEMM_CASE(AMN, BMN)                                                    \
    if (c_dtype == VELORA_BF16) { VELORA_GEMM_WIDTH(AMN, BMN, __nv_bfloat16) }       \
    VELORA_GEMM_WIDTH(AMN, BMN, float)
    if (!a_mn && !b_mn) { VELORA_GEMM_CASE(false, false) }
    if (!a_mn && b_mn) { VELORA_GEMM_CASE(false, true) }
    VELORA_GEMM_CASE(true, true)
#undef VELORA_GEMM_CASE
#undef VELORA_GEMM_WIDTH
}

int launch_linear_forward_tc(const void* X, int64_t ldx, const void* W, int64_t ldw, const float* v,
                             void* Y, int64_t ldy, void* Z, int z_dtype, int64_t ldz,
                             int dtype, int64_t N, int64_t D, int64_t O, int Dsub, int* status, cudaStream_t stream)
{
    // Fused path: Dsub a power of two between 8 and 1024 (sub-token boundaries then fall on 16-byte
    // chunks of the 64-column X tiles); everything else runs the GEMM and the compress kernel in turn.
    if (dtype == VELORA_BF16 && O <= 64) {               // adapter-shaped: one pass over X for Y and Z
        const int src = launch_linear_forward_skinny(X, ldx, W, ldw, v, Y, ldy, Z, z_dtype, ldz, N, D, O, Dsub, status, stream);
        if (src != VELORA_ERR_UNSUPPORTED) return src;
    }
    const bool pow2 = Dsub >= 8 && Dsub <= VELORA_MAX_DSUB && (Dsub & (Dsub - 1)) == 0;
    const bool gemm_ok = dtype == VELORA_BF16 && N >= 1 && N < (1 << 30) && D < (1 << 30) && O < (1 << 30) &&
                         tc_operand_ok(X, ldx) && tc_operand_ok(W, ldw);
    // A CTA compresses one tiles_n-th of its row block's columns while it multiplies all of them; the loads and
    // shuffles of that compete with the tensor cores' operand stream, so with few n-tiles the two kernels in turn are
    // faster.  Fused / in turn, us: 47 / 34 at 8192 x 1376 -> 1024 (4 n-tiles), 59 / 62 at 4096 x 4096 -> 2048 (8), 98 / 93
    // there with D = 5461 and a pitch of 10928 bytes (each load touches a line more), 51 / 58 at 12608 x 768 -> 3072 (12).
    const bool wide = (O + 255) / 256 >= (ldx % 64 == 0 ? 8 : 12);
    if (pow2 && gemm_ok && wide) {
        DeviceInfo di;
        int rc = device_info(&di);
        if (rc != VELORA_OK) return rc;
        GemmShape shape = gemm_shape(N, O, D, di.sm_count, true);
        if (shape.pair) {
            const int prc = launch_linear_forward_tc_pair(X, ldx, W, ldw, v, Y, ldy, Z, z_dtype, ldz, N, D, O, Dsub, status, stream);
            if (prc != VELORA_ERR_UNSUPPORTED) return prc;
            shape = GemmShape{false, 256, 1};
        }
        return launch_linear_forward_tc_single(shape, X, ldx, W, ldw, v, Y, ldy, Z, z_dtype, ldz, N, D, O, Dsub, status, stream);
    }
    int rc = launch_gemm_tc(GEMM_NT_K_K, X, ldx, W, ldw, Y, dtype, ldy, 0, N, O, D, dtype, status, stream);
    if (rc != VELORA_OK) return rc;
    return launch_compress(X, dtype, N, D, ldx, Dsub, v, Z, z_dtype, ldz, stream);
}

}  // namespace velora
