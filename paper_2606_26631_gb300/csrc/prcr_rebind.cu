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
// at v + D/2 (the rotate-half partners), for K and V, and walks the G layers
// two at a time. Consecutive threads cover consecutive 16-byte vectors of a
// row, so every warp-wide load and store is a set of whole 128-byte lines.
//
// HBM-bound. The first two layers' loads go out before the cos/sin, whose
// latency they hide: measured 16 sequences x 4 x 640 tokens x 36 layers x 8
// heads of 128 (11.5 GB) 1689 -> 1684 us (6.83 TB/s), 8 x ~512 x 28 x 4 (0.47
// GB) 84.0 -> 82.1 us, the smaller ones mostly from their layer groups. One
// layer ahead of the one stored instead (72 registers): 97 us for the second.
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
// of which the lookups here leave a few. Only the first wave's CTAs are there by
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
    for (int t = warp; t < a.tok_per_cta; t += nw) {
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

__global__ void __launch_bounds__(512) rebind_kernel(const __grid_constant__ RebindArgs a) {
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
    const uint16_t* sk = a.store_k + s_off;
    const uint16_t* sv = a.store_v + s_off;
    // two layers' vectors (K and its rotate-half partner, V likewise), the
    // first two requested before the cos/sin
    uint4 x[2][4];
    auto load = [&](int n) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (u < n) {
                x[u][0] = ld_stream(sk + u * sls);
                x[u][1] = ld_stream(sk + u * sls + P);
                x[u][2] = ld_stream(sv + u * sls);
                x[u][3] = ld_stream(sv + u * sls + P);
            }
        }
    };
    if (dst >= 0) load(l1 - l0);

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
    uint16_t* ck = a.cache_k + dst + int64_t(l0) * cls + off;
    uint16_t* cv = a.cache_v + dst + int64_t(l0) * cls + off;
    for (int l = l0; l < l1; l += 2) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (l + u < l1) {
                uint4 o0, o1;
                rotate_vec(x[u][0], x[u][1], c, s, o0, o1);
                st_row(ck + u * cls, o0);
                st_row(ck + u * cls + P, o1);
                st_row(cv + u * cls, x[u][2]);
                st_row(cv + u * cls + P, x[u][3]);
            }
        }
        sk += 2 * sls; sv += 2 * sls; ck += 2 * cls; cv += 2 * cls;
        load(l1 - l - 2);
    }
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
