// Prefill capture kernel (Sec. 3.1, Eq. "raw_kv" and "global_raw_memory",
// with the position-bound cache entry of Eq. "historical_position_bound_kv").
//
// During multimodal prefill each visual token's pre-rotation key and value
// rows exist once, per layer. This kernel reads them once and writes them
// twice: unchanged into the raw visual memory (with the token's original
// (t, h, w) coordinate), and as the ordinary decoder-cache entry the model
// itself would store: the key rotated with M-RoPE at the original
// coordinate, the value unchanged, at consecutive cache slots.
//
// Work layout as in the rebind kernel: a CTA owns T tokens x G layers; its
// prologue resolves each token's cache row (block-table lookup for paged
// caches) and the float32 cos/sin of every (token, pair) from the angle
// reduced modulo a turn in fixed point; each thread then owns one (token, head, 16-byte
// vector) and its rotate-half partner, for all G layers.
//
// HBM-bound (2 rows read, 4 written per token, layer and KV head). A layer's
// four vectors are requested one layer ahead, the first before the prologue,
// whose sin/cos and block-table latency they hide; the kernel is launched
// programmatically, so a prefill's calls, one per sequence, follow each other
// without a launch gap. Measured: 8 images of
// 2116 tokens x 28 layers x 4 heads (2.9 GB, 8 calls) 558 -> 465 us (6.3 TB/s);
// 3 of 768 x 36 x 8 189 -> 157 us; one of 8192 545 -> 527 us (6.9 TB/s). Held to
// 64 registers (four CTAs per SM) 557 us.
#include "prcr_device.cuh"
#include "prcr_pdl.cuh"

namespace prcr {
namespace {

template <int THREADS, int CTAS, bool AHEAD>
__global__ void __launch_bounds__(THREADS, CTAS) capture_kernel(const __grid_constant__ CaptureArgs a) {
    extern __shared__ __align__(16) float smem[];
    const int D = a.head_dim;
    const int P = D >> 1;
    const int T = a.tok_per_cta;
    float* cos_s = smem;
    float* sin_s = smem + T * P;
    int64_t* dst_s = reinterpret_cast<int64_t*>(sin_s + T * P);
    const int tok0 = blockIdx.x * T;
    uint32_t err = 0;

    // this thread's (token, head, 16-byte vector) and its rows
    const int lanes = a.lanes;
    const int my_t = threadIdx.x / lanes;
    const int lane = threadIdx.x - my_t * lanes;
    const int my_j = tok0 + my_t;
    const bool act = my_t < T && my_j < a.m_count;
    const int vph = D >> 4;
    const int h = lane / vph;
    const int v = lane - h * vph;
    const int64_t off = int64_t(h) * D + v * 8;
    const int l0 = blockIdx.y * a.layers_per_cta;
    const int l1 = min(l0 + a.layers_per_cta, a.n_layers);
    const int64_t s_off = int64_t(l0) * a.src_layer_stride + int64_t(my_j) * a.src_token_stride + off;
    const uint16_t* sk = a.src_k + s_off;
    const uint16_t* sv = a.src_v + s_off;
    uint4 k0, k1, v0, v1;
    auto load = [&]() {
        k0 = ld_stream(sk);
        k1 = ld_stream(sk + P);
        v0 = ld_stream(sv);
        v1 = ld_stream(sv + P);
    };
    pdl_allow();
    pdl_wait();
    if (AHEAD && act) load();

    for (int t = threadIdx.x; t < T; t += blockDim.x) {
        const int j = tok0 + t;
        int64_t dst = -1;
        if (j < a.m_count) {
            const int64_t slot = a.slot_begin + j;
            if (slot >= a.capacity) {
                err |= PRCR_ST_CAPACITY;
            } else if (a.cache_kind == PRCR_CACHE_CONTIGUOUS) {
                dst = a.cache_seq_off + slot * a.slot_stride;
            } else {
                const int64_t lb = slot / a.block_size;
                const int32_t blk = a.bt_row[lb];
                if (blk < 0 || blk >= a.n_blocks) err |= PRCR_ST_NO_BLOCK;
                else dst = int64_t(blk) * a.block_stride + (slot - lb * a.block_size) * a.slot_stride;
            }
            if (a.store_coords && blockIdx.y == 0) {
                a.store_coords[3 * int64_t(j) + 0] = a.coords[3 * int64_t(j) + 0];
                a.store_coords[3 * int64_t(j) + 1] = a.coords[3 * int64_t(j) + 1];
                a.store_coords[3 * int64_t(j) + 2] = a.coords[3 * int64_t(j) + 2];
            }
        }
        dst_s[t] = dst;
    }
    for (int q = threadIdx.x; q < T * P; q += blockDim.x) {
        const int t = q / P;
        const int i = q - t * P;
        const int j = tok0 + t;
        float c = 1.0f, s = 0.0f;
        if (j < a.m_count) {
            const int ax = pair_axis(i, a.layout, a.sec_t, a.sec_h, a.sec_w);
            sincos_turns(double(a.coords[3 * int64_t(j) + ax]), a.turn_freq[i], &s, &c);
        }
        cos_s[q] = c;
        sin_s[q] = s;
    }
    if (err && blockIdx.y == 0) atomicOr(a.status, err);
    __syncthreads();

    if (!act) return;
    const int64_t dst = dst_s[my_t];
    float c[8], s[8];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const float4 c4 = *reinterpret_cast<const float4*>(cos_s + my_t * P + v * 8 + 4 * u);
        const float4 s4 = *reinterpret_cast<const float4*>(sin_s + my_t * P + v * 8 + 4 * u);
        c[4 * u] = c4.x; c[4 * u + 1] = c4.y; c[4 * u + 2] = c4.z; c[4 * u + 3] = c4.w;
        s[4 * u] = s4.x; s[4 * u + 1] = s4.y; s[4 * u + 2] = s4.z; s[4 * u + 3] = s4.w;
    }
    const int64_t r_off = int64_t(l0) * a.store_layer_stride + int64_t(my_j) * a.store_token_stride + off;
    uint16_t* rk = a.store_k + r_off;
    uint16_t* rv = a.store_v + r_off;
    const int64_t c_off = (dst < 0 ? 0 : dst) + int64_t(l0) * a.cache_layer_stride + off;  // never written if dst < 0
    uint16_t* ck = a.cache_k + c_off;
    uint16_t* cv = a.cache_v + c_off;
    for (int l = l0; l < l1; ++l) {
        if (!AHEAD) load();
        const uint4 x0 = k0, x1 = k1, y0 = v0, y1 = v1;
        sk += a.src_layer_stride;
        sv += a.src_layer_stride;
        if (AHEAD && l + 1 < l1) load();
        st_row(rk, x0);
        st_row(rk + P, x1);
        st_row(rv, y0);
        st_row(rv + P, y1);
        if (dst >= 0) {
            uint4 o0, o1;
            rotate_vec(x0, x1, c, s, o0, o1);
            st_row(ck, o0);
            st_row(ck + P, o1);
            st_row(cv, y0);
            st_row(cv + P, y1);
        }
        rk += a.store_layer_stride; rv += a.store_layer_stride;
        ck += a.cache_layer_stride; cv += a.cache_layer_stride;
    }
}

}  // namespace

namespace {

// Rows of more than 384 threads (n_kv_heads x head_dim > 6144): without a layer
// ahead, in 64 registers, or the CTA is alone on its SM. 64 heads of 128, 2 images of 5920 tokens x 2 layers 402
// -> 350 us, one of 1600 x 24 605 -> 554; up to 384 threads two CTAs fit as they are.
using CaptureKernel = void (*)(CaptureArgs);
CaptureKernel capture_for(int block) { return block > 384 ? capture_kernel<512, 2, false> : capture_kernel<384, 1, true>; }

}  // namespace

cudaError_t capture_blocks_per_sm(int block, size_t smem, int* out) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, capture_for(block), block, smem);
}

cudaError_t launch_capture(const CaptureArgs& a, dim3 grid, int block, size_t smem,
                           cudaStream_t stream) {
    return launch_pdl(capture_for(block), grid, dim3(unsigned(block)), smem, stream, a);
}

}  // namespace prcr
