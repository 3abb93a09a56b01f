// Rows that TMA cannot address, copied to rows that it can.
//
// A tensor map wants a 16-byte aligned base and a row pitch that is a multiple of 16 bytes; a bf16 matrix as a
// framework allocates it (5461 columns, no padding) has neither.  Such an operand is copied once into the
// workspace and the tensor-core kernels run on the copy.  The copy is one read and one write of the operand; without
// it the product runs on the CUDA cores.  The copy's pitch is a multiple of 128 bytes, not of the 16 that TMA asks for:
// a 4096 x 5461 -> 2048 product took 84 us with both operands at a pitch of 10928 bytes (every other row starts in
// the middle of a 32-byte sector) and 70 us at 11008.
//
// A warp takes 128 consecutive 16-byte chunks of a row, four per lane, all loads issued before the first is used.
// The source of a chunk sits at any even byte offset, the same for a whole row.  A lane loads the aligned 16 bytes in which
// its chunk begins, takes the rest from its neighbour (whose chunk begins there) and shifts; only the last lane of the
// last step loads a second time.
#include "gemm_tc.cuh"
#include "row_chunks.cuh"

namespace velora {
namespace {

constexpr int PK_THREADS = 256;
constexpr int PK_U = 4;                                    // chunks per lane
constexpr int PK_SEG = 32 * PK_U;                          // chunks per warp and step

struct PackArgs {
    const char* src[2];
    const char* src_end[2];                                // one past the last element
    int64_t src_pitch[2];                                  // bytes
    uint4* dst[2];
    int64_t dst_pitch[2];                                  // chunks
    int chunks[2], segs[2];
    int64_t items[2];                                      // rows x segments
};

__global__ void __launch_bounds__(PK_THREADS)
pack_rows_kernel(const PackArgs a)
{
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (PK_THREADS / 32);
    const int64_t total = a.items[0] + a.items[1];
    for (int64_t it = static_cast<int64_t>(blockIdx.x) * (PK_THREADS / 32) + (threadIdx.x >> 5); it < total; it += warps) {
        const int k = it < a.items[0] ? 0 : 1;
        const unsigned item = static_cast<unsigned>(it - (k ? a.items[0] : 0));
        const unsigned row = item / static_cast<unsigned>(a.segs[k]);
        const int c0 = static_cast<int>(item - row * a.segs[k]) * PK_SEG + lane;
        const char* rp = a.src[k] + static_cast<int64_t>(row) * a.src_pitch[k];
        const uint32_t shift = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(rp) & 15u);
        const char* ap = rp - shift;
        uint4 d[PK_U], over = make_uint4(0u, 0u, 0u, 0u);     // chunks at or beyond the row's end are loaded, not used
#pragma unroll
        for (int u = 0; u < PK_U; ++u)
            d[u] = c0 - lane + 32 * u <= a.chunks[k] ? load_aligned_chunk(ap + 16 * static_cast<int64_t>(c0 + 32 * u), a.src[k], a.src_end[k])
                                                     : make_uint4(0u, 0u, 0u, 0u);
        if (lane == 31) over = load_aligned_chunk(ap + 16 * static_cast<int64_t>(c0 + 32 * PK_U - 31), a.src[k], a.src_end[k]);
        over.x = __shfl_sync(0xffffffffu, over.x, 31); over.y = __shfl_sync(0xffffffffu, over.y, 31);
        over.z = __shfl_sync(0xffffffffu, over.z, 31); over.w = __shfl_sync(0xffffffffu, over.w, 31);
        uint4* op = a.dst[k] + static_cast<int64_t>(row) * a.dst_pitch[k];
#pragma unroll
        for (int u = 0; u < PK_U; ++u) {
            // The next chunk's beginning: lane + 1 of this step, for lane 31 lane 0 of the next.
            const uint4 nx = u + 1 < PK_U ? d[(u + 1) % PK_U] : over;
            const uint4 give = lane == 0 ? nx : d[u];
            const int from = (lane + 1) & 31;
            uint4 y;
            y.x = __shfl_sync(0xffffffffu, give.x, from); y.y = __shfl_sync(0xffffffffu, give.y, from);
            y.z = __shfl_sync(0xffffffffu, give.z, from); y.w = __shfl_sync(0xffffffffu, give.w, from);
            if (c0 + 32 * u < a.chunks[k]) op[c0 + 32 * u] = shift_chunks(d[u], y, shift);
        }
    }
}

}  // namespace

int64_t pack_rows_pitch(int64_t cols) { return (cols + 63) / 64 * 64; }

size_t pack_rows_bytes(int64_t rows, int64_t cols)
{
    return (static_cast<size_t>(rows) * static_cast<size_t>(pack_rows_pitch(cols)) * 2 + 255) / 256 * 256;
}

int launch_pack_rows(const PackJob* jobs, int count, cudaStream_t stream)
{
    PackArgs a{};
    for (int k = 0; k < count && k < 2; ++k) {
        const PackJob& j = jobs[k];
        if (j.rows < 1 || j.rows >= (1 << 30) || j.cols < 1 || j.cols >= (1 << 30)) return VELORA_ERR_UNSUPPORTED;
        a.src[k] = static_cast<const char*>(j.src);
        a.src_pitch[k] = j.ld * 2;
        a.src_end[k] = a.src[k] + ((j.rows - 1) * j.ld + j.cols) * 2;
        a.dst[k] = static_cast<uint4*>(j.dst);
        a.chunks[k] = static_cast<int>((j.cols + 7) / 8);
        a.dst_pitch[k] = pack_rows_pitch(j.cols) / 8;
        a.segs[k] = (a.chunks[k] + PK_SEG - 1) / PK_SEG;
        a.items[k] = j.rows * a.segs[k];
        if (a.items[k] >= (static_cast<int64_t>(1) << 31)) return VELORA_ERR_UNSUPPORTED;
    }
    const int64_t items = a.items[0] + a.items[1];
    if (items == 0) return VELORA_OK;
    DeviceInfo di;
    const int rc = device_info(&di);
    if (rc != VELORA_OK) return rc;
    int64_t grid = ceil_div64(items, PK_THREADS / 32);
    const int64_t cap = static_cast<int64_t>(di.sm_count) * kStreamCtasPerSm;
    if (grid > cap) grid = cap;
    return launch_chained(pack_rows_kernel, dim3(static_cast<unsigned>(grid)), PK_THREADS, 0, stream, a);
}

}  // namespace velora
