// Raw visual memory fill (Sec. 3.1, Eq. "raw_kv" and "global_raw_memory"):
// a strided, 16-byte vectorised copy of pre-rotation K/V rows and of the
// tokens' original coordinates into the store.
//
// HBM-bound. A CTA copies kPer x 256 vectors of K and of V of one layer, all of
// a thread's loads requested before its first store; rows are found with one
// 32-bit division per vector, and with none where both sides' tokens follow
// each other without gaps (FLAT: a layer is then one run). Measured:
// 2116 tokens x 28 layers x 4 heads of 128 (243 MB) 41.5 -> 36.5 us (6.66
// TB/s), 2 x 8192 x 36 x 8 723 -> 686 us (7.05 TB/s); before, one vector of
// each at a time in a grid-stride loop with two 64-bit divisions.
#include "prcr_device.cuh"
#include "prcr_pdl.cuh"

namespace prcr {
namespace {

constexpr int kThreads = 256;
constexpr int kPer = 4;  // vectors of K and of V per thread

template <bool FLAT>
__global__ void __launch_bounds__(kThreads) store_kernel(const __grid_constant__ StoreArgs a) {
    pdl_allow();
    pdl_wait();
    const int64_t n = int64_t(a.m_count) * a.row_vecs;  // vectors of a layer
    const int64_t i0 = int64_t(blockIdx.x) * (kThreads * kPer) + threadIdx.x;
    for (int l = blockIdx.y; l < a.n_layers; l += gridDim.y) {
        const uint16_t* sk = a.src_k + l * a.src_layer_stride;
        const uint16_t* sv = a.src_v + l * a.src_layer_stride;
        const int64_t dl = l * a.dst_layer_stride;
        uint4 k[kPer], v[kPer];
        int64_t d[kPer];
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int64_t i = i0 + u * kThreads;
            if (i >= n) continue;
            int64_t so = 8 * i;
            d[u] = so;
            if (!FLAT) {
                const int64_t m = n <= INT32_MAX ? int64_t(uint32_t(i) / uint32_t(a.row_vecs)) : i / a.row_vecs;
                const int64_t e = 8 * (i - m * a.row_vecs);
                so = m * a.src_token_stride + e;
                d[u] = m * a.dst_token_stride + e;
            }
            k[u] = ld_stream(sk + so);
            v[u] = ld_stream(sv + so);
        }
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            if (i0 + u * kThreads >= n) continue;
            st_row(a.dst_k + dl + d[u], k[u]);
            st_row(a.dst_v + dl + d[u], v[u]);
        }
    }
    if (a.dst_coords && blockIdx.y == 0) {
        for (int64_t i = int64_t(blockIdx.x) * kThreads + threadIdx.x; i < 3 * int64_t(a.m_count);
             i += int64_t(gridDim.x) * kThreads)
            a.dst_coords[i] = a.src_coords[i];
    }
}

}  // namespace

cudaError_t launch_store(const StoreArgs& a, cudaStream_t stream) {
    const int64_t n = int64_t(a.m_count) * a.row_vecs;
    const int64_t row = 8 * int64_t(a.row_vecs);
    const dim3 grid(unsigned((n + kThreads * kPer - 1) / (kThreads * kPer)),
                    unsigned(a.n_layers < 65535 ? a.n_layers : 65535), 1);
    const bool flat = a.m_count == 1 || (a.src_token_stride == row && a.dst_token_stride == row);
    return flat ? launch_pdl(store_kernel<true>, grid, dim3(kThreads), 0, stream, a)
                : launch_pdl(store_kernel<false>, grid, dim3(kThreads), 0, stream, a);
}

}  // namespace prcr
