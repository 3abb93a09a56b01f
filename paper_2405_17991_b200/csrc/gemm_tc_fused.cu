// The forward with compress riding on it (gemm_fuse.cuh), single-CTA shapes.
#include "gemm_tc_kernel.cuh"

namespace velora {

int launch_linear_forward_tc_single(const GemmShape& shape, const void* X, int64_t ldx, const void* W, int64_t ldw, const float* v,
                                    void* Y, int64_t ldy, void* Z, int z_dtype, int64_t ldz,
                                    int64_t N, int64_t D, int64_t O, int Dsub, int* status, cudaStream_t stream)
{
    CUtensorMap ta, tb;
    int rc = make_tmap_bf16_2d(&ta, X, D, N, ldx, BK, BM);
    if (rc != VELORA_OK) return rc;
    rc = make_tmap_bf16_2d(&tb, W, D, O, ldw, BK, shape.bn);
    if (rc != VELORA_OK) return rc;
    const FuseArgs fz{v, Z, ldz, Dsub, static_cast<int>(ceil_div64(D, Dsub)), static_cast<const uint4*>(X), ldx / 8};
    const int m = static_cast<int>(N), n = static_cast<int>(O), k = static_cast<int>(D);
#define VELORA_FUSED_CASE(ZK)                                                                                                            \
    return shape.bn == 128                                                                                                               \
               ? launch_kernel<false, false, __nv_bfloat16, ZK, 128>(ta, tb, Y, ldy, 0, m, n, k, shape.splits, status, stream, fz)       \
               : launch_kernel<false, false, __nv_bfloat16, ZK, 256>(ta, tb, Y, ldy, 0, m, n, k, shape.splits, status, stream, fz)
    if (z_dtype == VELORA_F32) { VELORA_FUSED_CASE(1); }
    if (z_dtype == VELORA_FP8_E4M3) { VELORA_FUSED_CASE(3); }
    VELORA_FUSED_CASE(2);
#undef VELORA_FUSED_CASE
}

}  // namespace velora
