// Rebind + inject kernel (Sec. 3.3, Eq. "cache_reconstruction" and
// "active_cache"; Algorithm 1, the loop over layers).
//
// For every selected token, every layer and every KV head, the raw key row
// is gathered from the store, rotated with M-RoPE at the token's reassigned
// (t, h, w) position, rounded to bf16 and written to the token's cache slot;
// the raw value row is copied unchanged next to it.
//
// Work layout. A CTA owns T tokens x G layers. Its threads first build the
// float32 cos/sin of every (token, rotation pair) of the tile in shared
// memory, once for all G layers and all heads: the angle modulo a turn is
// formed exactly in fixed-point integers (sincos_turns) and only then handed
// to float32 sincosf, so a position near 3e4 keeps a ~2e-7 rad angle error
// instead of the ~2e-3 of a float32 product.
// Each thread owns one (token, head, 16-byte vector v) slot of the row: it
// loads the 8 bf16 of the first half at v and the 8 bf16 of the second half
// at v + D/2 (the rotate-half partners), for K and V, and walks the G
// layers, two in flight. Consecutive threads cover consecutive 16-byte vectors of a
// row, so every warp-wide load and store is a set of whole 128-byte lines.
//
// HBM-bound where there are many rows. The first layer's loads go out before the
// cos/sin, whose latency they hide. 64 registers, four CTAs of 256 threads per SM:
// with two layers requested ahead (75 registers, three CTAs) few heads or few layers,
// whose cos/sin weigh most, were slower than with none. Whole revisits in us, no
// layer ahead | two | one (each with its own rule for the groups of layers, the last
// stream_layers_per_cta's): 8 sequences x ~512 tokens x 28 layers x 4 heads of 128
// (0.47 GB) 84.4 | 81.5 | 80.5, 3 x ~650 x 6 x 8 14.3 | 16.0 | 13.1, 3 x ~3700 x 5 x 3
// 19.4 | 23.7 | 17.9, 9 x ~320 x 21 x 1 of 256 33.3 | 43.9 | 29.2; 16 x 4 x 640 x 36 x
// 8 (11.5 GB) 1684 | 1680 | 1674 (6.9 TB/s).
//
// The kernel is launched with programmatic dependent launch behind the plan
// kernel and waits on it (griddepcontrol.wait) before touching the plan; its
// first rows are prefetched into L2 meanwhile (prefetch_rows).
#include "prcr_device.cuh"
#include "prcr_pdl.cuh"

namespace prcr {
namespace {

constexpr int kEarlyLayers = 4;

// The raw rows of the CTA's tokens (its first kEarlyLayers layers) into L2 while
// the plan kernel of the same call runs (which releases this one when all before
// the call is done; behind any other kernel nothing is read before the wait).
// Hints only: nothing read here is used for anything else, so indices or offsets
// that are wrong cost time alone; what is prefetched lies in the store whatever
// they hold. The plan takes ~8 us,
// of which the lookups here, three dependent loads a token, leave a few: two tokens a
// warp at most (a CTA of few short heads has up to 256 tokens, and all of them made 9
// sequences x ~290 tokens x 21 layers x 3 heads of 16 12.8 -> 16.2 us, 12 x ~600 x 8 x
// 1 of 32 16.5 -> 25.8; now 13.3 and 15.2). Only the first wave's CTAs are there by
// then. Measured (calls in a row, without | 2 layers | 4 | 12): 3 x 267 tokens x 8
// layers x 8 heads of 128 32.2 | 31.9 | 31.1 | 31.1 us, 5 x 443 x 32 x 5 41.2 | 40.6
// | 39.9 | 39.9, 12 x 201 x 11 x 5 of 256 49.9 | 49.9 | 49.0 | 49.0, 8 x ~512 x 28
// x 4 81.6 | 82.1 | 81.5 | 81.5.
__device__ __forceinline__ void prefetch_rows(const RebindArgs& a) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = int(blockDim.x + 31) >> 5;
    if ((blockDim.x & 31) && warp == nw - 1) return;  // a part of a warp
    const int l = int(blockIdx.y) * a.layers_per_cta + (lane >> 1);
    const int n = min(kEarlyLayers, a.layers_per_cta);
    const uint32_t bytes = uint32_t(a.lanes) * 32;  // of a row
    for (int t = warp; t < min(a.tok_per_cta, 2 * nw); t += nw) {
        const int64_t j = int64_t(blockIdx.x) * a.tok_per_cta + t;
        if (j >= a.total_k) break;
        const int m = a.idx[j];
        const int b = sequence_of(a.seq_rev_off, a.n_seqs, sequence_of(a.rev_tok_off, a.n_revisits, int(j)));
        if (m < 0 || m >= a.n_tokens || (lane >> 1) >= n || l >= a.n_layers) continue;
        const uint16_t* row = (lane & 1 ? a.store_v : a.store_k) + b * a.store_seq_stride +
                              int64_t(l) * a.store_layer_stride + int64_t(m) * a.store_token_stride;
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(row), "r"(bytes) : "memory");
    }
}

__global__ void __launch_bounds__(512, 2) rebind_kernel(const __grid_constant__ RebindArgs a) {
    extern __shared__ __align__(16) float smem[];
    pdl_allow();
    if (int64_t(blockIdx.y) * gridDim.x + blockIdx.x < a.early_ctas) prefetch_rows(a);
    pdl_wait();
    if (*reinterpret_cast<const volatile uint32_t*>(a.status) & PRCR_ST_CSR) return;

    const int D = a.head_dim;
    const int P = D >> 1;
    const int T = a.tok_per_cta;
    float* cos_s = smem;
    float* sin_s = smem + T * P;
    const int64_t tok0 = int64_t(blockIdx.x) * T;

    const int lanes = a.lanes;
    const int my_t = threadIdx.x / lanes;
    const int lane = threadIdx.x - my_t * lanes;
    const int64_t my_tok = tok0 + my_t;
    const int64_t dst = my_t < T && my_tok < a.total_k ? a.plan_dst[my_tok] : -1;
    const int vph = D >> 4;  // 16-byte vectors per half row of one head
    const int h = lane / vph;
    const int v = lane - h * vph;
    const int64_t off = int64_t(h) * D + v * 8;
    const int l0 = blockIdx.y * a.layers_per_cta;
    const int l1 = min(l0 + a.layers_per_cta, a.n_layers);
    const int64_t sls = a.store_layer_stride;
    const int64_t cls = a.cache_layer_stride;
    const int64_t s_off = (dst < 0 ? 0 : a.plan_src[my_tok]) + int64_t(l0) * sls + off;
    // the first layer's vectors (K and its rotate-half partner, V likewise),
    // requested before the cos/sin
    uint4 x[4];
    if (dst >= 0) {
        x[0] = ld_stream(a.store_k + s_off);
        x[1] = ld_stream(a.store_k + s_off + P);
        x[2] = ld_stream(a.store_v + s_off);
        x[3] = ld_stream(a.store_v + s_off + P);
    }

    for (int q = threadIdx.x; q < T * P; q += blockDim.x) {
        const int t = q / P;
        const int i = q - t * P;
        const int64_t tok = tok0 + t;
        float c = 1.0f, s = 0.0f;
        if (tok < a.total_k) {
            const int ax = pair_axis(i, a.layout, a.sec_t, a.sec_h, a.sec_w);
            sincos_turns(a.plan_pos[3 * tok + ax], a.turn_freq[i], &s, &c);
        }
        cos_s[q] = c;
        sin_s[q] = s;
    }
    __syncthreads();
    if (dst < 0) return;

    float c[8], s[8];
    {
        const float4* cp = reinterpret_cast<const float4*>(cos_s + my_t * P + v * 8);
        const float4* sp = reinterpret_cast<const float4*>(sin_s + my_t * P + v * 8);
        const float4 c0 = cp[0], c1 = cp[1], s0 = sp[0], s1 = sp[1];
        c[0] = c0.x; c[1] = c0.y; c[2] = c0.z; c[3] = c0.w;
        c[4] = c1.x; c[5] = c1.y; c[6] = c1.z; c[7] = c1.w;
        s[0] = s0.x; s[1] = s0.y; s[2] = s0.z; s[3] = s0.w;
        s[4] = s1.x; s[5] = s1.y; s[6] = s1.z; s[7] = s1.w;
    }
    const int64_t c_off = dst + int64_t(l0) * cls + off;
    uint16_t* ck = a.cache_k + c_off;
    uint16_t* cv = a.cache_v + c_off;
    uint4 o0, o1;
    rotate_vec(x[0], x[1], c, s, o0, o1);
    st_row(ck, o0);
    st_row(ck + P, o1);
    st_row(cv, x[2]);
    st_row(cv + P, x[3]);
    stream_layers(a.store_k + s_off + sls, a.store_v + s_off + sls, ck + cls, cv + cls, sls, cls, P, l1 - l0 - 1, c, s);
}

}  // namespace

cudaError_t rebind_blocks_per_sm(int block, size_t smem, int* out) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, rebind_kernel, block, smem);
}

cudaError_t launch_rebind(const RebindArgs& a, dim3 grid, int block, size_t smem,
                          cudaStream_t stream) {
    return launch_pdl(rebind_kernel, grid, dim3(unsigned(block)), smem, stream, a);
}

}  // namespace prcr
