// The selection's steps after the logits, on clusters of CTAs, one cluster per
// sequence.
//
// Rank r of a cluster of C CTAs takes the tokens r * T .. r * T + T - 1 of its
// sequence (T = tok_per_cta). Two exchanges through distributed shared memory
// stand where kernel boundaries would:
//   1. softmax statistics: every CTA reduces its tokens' logits to a (max, sum
//      of exp) per query head; after a cluster barrier each CTA merges all C
//      of them into the heads' normalisers;
//   2. relevance of the CTA's own tokens (mean over the heads of the softmax
//      weight, heads in ascending order), left in shared memory; after a
//      second barrier each CTA copies the whole sequence's relevances.
// Every CTA then finds the K-th largest relevance by itself (the same answer
// in each) and writes its own tokens' share of the selection in index order,
// knowing from the copy how many lie before its first token. The search
// narrows the range of float bits (relevance >= 0, so bit order is value
// order) that holds the K-th largest: 2048 buckets spread over the range from
// the smallest to the largest relevance, counted by shared-memory atomics
// (about M / 2048 keys meet in a bucket), then the few keys of its bucket
// ranked by one warp; or again over that bucket while it holds many.
#include <array>
#include <cmath>
#include <map>
#include <mutex>
#include <utility>

#include "prcr_pdl.cuh"
#include "prcr_select.cuh"

namespace prcr {
namespace {

constexpr int kMaxCluster = 16;
constexpr int kBuckets = 2048;
constexpr unsigned kAll = 0xffffffffu;

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Address of this CTA's shared variable at `p` in the shared memory of CTA
// `rank` of the cluster, and loads from there.
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(r)
                 : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
    return r;
}
__device__ __forceinline__ float2 peer_f32x2(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint4 peer_u32x4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(addr));
    return v;
}

// What the phases share, in static shared memory.
struct SelectShared {
    float2 stat[kSelectMaxQHeads];  // this CTA's (max, sum) per query head; read by the peers
    float2 norm[kSelectMaxQHeads];  // (max, 1 / (sum * n_q_heads)) over the whole sequence
    uint32_t hist[kBuckets];
    uint2 range;                    // smallest and largest key of this CTA's tokens; read by the peers
    uint32_t wsum[32];              // per warp: keys in its buckets; later equal | above << 16 in its tokens
    uint32_t before[2][32];         // per warp: keys equal to X and above it before this CTA's first token
    uint32_t pick[3];               // bucket of the K-th largest, keys in it, keys above it
    uint32_t list[32], n_list;
};

// Exchange 1: the heads' normalisers from every CTA's statistics. Also
// sets up the search's shared state.
template <int NT>
__device__ __forceinline__ void merge_stats(const SelectArgs& a, int C, SelectShared& sh) {
    cluster_arrive();
    for (int i = threadIdx.x; i < kBuckets; i += NT) sh.hist[i] = 0u;
    if (threadIdx.x == 0) {
        sh.range = make_uint2(0xffffffffu, 0u);
        sh.n_list = 0u;
    }
    cluster_wait();
    const int c = threadIdx.x & (kMaxCluster - 1);
    for (int h0 = 0; h0 < a.n_q_heads; h0 += NT / kMaxCluster) {
        const int hq = h0 + threadIdx.x / kMaxCluster;
        float2 v = make_float2(-INFINITY, 0.0f);
        if (hq < a.n_q_heads && c < C) v = peer_f32x2(peer_addr(&sh.stat[hq], uint32_t(c)));
        float m = v.x;
#pragma unroll
        for (int o = kMaxCluster / 2; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kAll, m, o));
        float z = v.x == -INFINITY ? 0.0f : v.y * __expf(v.x - m);
#pragma unroll
        for (int o = kMaxCluster / 2; o; o >>= 1) z += __shfl_xor_sync(kAll, z, o);
        // no finite logit (no readable token, or a query position out of
        // range): every weight of this head is taken as 0
        if (hq < a.n_q_heads && c == 0)
            sh.norm[hq] = m == -INFINITY ? make_float2(0.0f, 0.0f)
                                         : make_float2(m, 1.0f / (z * float(a.n_q_heads)));
    }
    __syncthreads();
}

// Exchange 2, the search and the output. keys [C * T] holds this CTA's own
// tokens' relevances at m_beg; the peers' are copied in. lo, hi: smallest and
// largest of the relevances that this thread wrote.
template <int NT>
__device__ __forceinline__ void select_topk(const SelectArgs& a, int b, int C, int m_beg, int nt, uint32_t* keys,
                                            uint32_t lo, uint32_t hi, SelectShared& sh) {
    constexpr int NW = NT / 32, BPT = kBuckets / NT;  // buckets per thread
    const int M = a.n_tokens, T = a.tok_per_cta;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    lo = __reduce_min_sync(kAll, lo);
    hi = __reduce_max_sync(kAll, hi);
    if (lane == 0 && lo <= hi) {
        atomicMin(&sh.range.x, lo);
        atomicMax(&sh.range.y, hi);
    }
    cluster_arrive();
    cluster_wait();
    uint2 range = make_uint2(0xffffffffu, 0u);
    if (lane < C) {
        const float2 v = peer_f32x2(peer_addr(&sh.range, uint32_t(lane)));
        range = make_uint2(__float_as_uint(v.x), __float_as_uint(v.y));
    }
#pragma unroll 4
    for (int i = 4 * tid; i < M; i += 4 * NT) {  // T is a multiple of 16: four tokens share a rank
        const int r = i / T;
        const uint4 v = peer_u32x4(peer_addr(keys + i, uint32_t(r)));
        if (r * T != m_beg) *reinterpret_cast<uint4*>(keys + i) = v;
    }
    cluster_arrive();  // this CTA has read its peers; it waits for their reads before it ends
    lo = __reduce_min_sync(kAll, range.x);
    hi = __reduce_max_sync(kAll, range.y);
    __syncthreads();

    // the K-th largest key X lies in [lo, hi]; `above` keys are larger than hi
    const uint32_t K = uint32_t(a.k);
    uint32_t above = 0u, X = lo;
    while (lo != hi) {  // the range shrinks by a factor of kBuckets / 2 at least
        const int bits = 32 - __clz(int(hi - lo));
        const int sh_b = max(0, bits - 11);
        for (int i = tid; i < M; i += NT) {
            const uint32_t k = keys[i];
            if (k >= lo && k <= hi) atomicAdd(&sh.hist[(k - lo) >> sh_b], 1u);
        }
        __syncthreads();
        // this thread's buckets, and the keys in higher ones (suffix sums)
        uint32_t cnt[BPT], mine = 0u;
#pragma unroll
        for (int u = 0; u < BPT; ++u) {
            cnt[u] = sh.hist[tid * BPT + u];
            sh.hist[tid * BPT + u] = 0u;  // for the next round
            mine += cnt[u];
        }
        uint32_t suf = mine;  // inclusive over the lanes above
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_down_sync(kAll, suf, o);
            if (lane + o < 32) suf += y;
        }
        if (lane == 0) sh.wsum[warp] = suf;
        __syncthreads();
        const uint32_t higher = __reduce_add_sync(kAll, lane > warp && lane < NW ? sh.wsum[lane] : 0u);
        uint32_t top = above + higher + suf - mine;  // keys above this thread's buckets
#pragma unroll
        for (int u = BPT - 1; u >= 0; --u) {
            if (top < K && top + cnt[u] >= K) {
                sh.pick[0] = uint32_t(tid * BPT + u);
                sh.pick[1] = cnt[u];
                sh.pick[2] = top;
            }
            top += cnt[u];
        }
        __syncthreads();
        const uint32_t n = sh.pick[1];
        lo += sh.pick[0] << sh_b;
        hi = min(hi, lo + ((1u << sh_b) - 1u));
        above = sh.pick[2];
        X = lo;
        if (sh_b == 0) break;
        if (above + n == K && lo > 0u) {  // the whole bucket is selected
            X = lo - 1u;
            above = K;
            break;
        }
        if (n <= 32u) {  // rank the bucket's keys
            for (int i = tid; i < M; i += NT) {
                const uint32_t k = keys[i];
                if (k >= lo && k <= hi) sh.list[atomicAdd(&sh.n_list, 1u)] = k;
            }
            __syncthreads();
            if (warp == 0) {
                const uint32_t v = lane < int(n) ? sh.list[lane] : 0u;
                uint32_t gt = 0u, ge = 0u;
                for (uint32_t j = 0; j < n; ++j) {
                    const uint32_t y = __shfl_sync(kAll, v, int(j));
                    gt += y > v ? 1u : 0u;
                    ge += y >= v ? 1u : 0u;
                }
                if (lane < int(n) && above + gt < K && above + ge >= K) {  // equal keys write the same
                    sh.pick[0] = v;
                    sh.pick[2] = above + gt;
                }
            }
            __syncthreads();
            X = sh.pick[0];
            above = sh.pick[2];
            break;
        }
        __syncthreads();  // pick is rewritten by the next round
    }

    // keys above X are all taken, and of those equal to X the first ones
    const uint32_t need_eq = K - above;
    const uint32_t below = (1u << lane) - 1u;
    uint32_t gt_b = 0u, eq_b = 0u;  // before this CTA's first token
    for (int i = tid; i < m_beg; i += NT) {
        const uint32_t k = keys[i];
        gt_b += k > X ? 1u : 0u;
        eq_b += k == X ? 1u : 0u;
    }
    gt_b = __reduce_add_sync(kAll, gt_b);
    eq_b = __reduce_add_sync(kAll, eq_b);
    // warp w takes a contiguous run of the CTA's tokens
    const int per = (nt + 32 * NW - 1) / (32 * NW) * 32, t_beg = warp * per, t_end = min(nt, t_beg + per);
    uint32_t gt_w = 0u, eq_w = 0u;
    for (int t = t_beg + lane; t < t_end; t += 32) {
        const uint32_t k = keys[m_beg + t];
        gt_w += k > X ? 1u : 0u;
        eq_w += k == X ? 1u : 0u;
    }
    gt_w = __reduce_add_sync(kAll, gt_w);
    eq_w = __reduce_add_sync(kAll, eq_w);
    if (lane == 0) {
        sh.before[0][warp] = eq_b;
        sh.before[1][warp] = gt_b;
        sh.wsum[warp] = eq_w | (gt_w << 16);  // at most 32768 tokens: no carry between the halves
    }
    __syncthreads();
    {
        const uint32_t w = lane < warp ? sh.wsum[lane] : 0u;
        uint32_t eq = __reduce_add_sync(kAll, (lane < NW ? sh.before[0][lane] : 0u) + (w & 0xffffu));
        uint32_t gt = __reduce_add_sync(kAll, (lane < NW ? sh.before[1][lane] : 0u) + (w >> 16));
        int32_t* dst = a.idx_out + int64_t(b) * a.k;
        for (int t0 = t_beg; t0 < t_end; t0 += 32) {
            const int t = t0 + lane;
            const uint32_t k = t < t_end ? keys[m_beg + t] : 0u;
            const bool is_eq = t < t_end && k == X, is_gt = t < t_end && k > X;
            const uint32_t beq = __ballot_sync(kAll, is_eq), bgt = __ballot_sync(kAll, is_gt);
            const uint32_t e = eq + uint32_t(__popc(beq & below));
            const uint32_t at = gt + uint32_t(__popc(bgt & below)) + min(e, need_eq);
            if ((is_gt || (is_eq && e < need_eq)) && at < K) dst[at] = m_beg + t;
            eq += uint32_t(__popc(beq));
            gt += uint32_t(__popc(bgt));
        }
    }
    if (m_beg == 0 && tid == 0) {
        a.rev_tok_off[b] = b * a.k;
        a.seq_rev_off[b] = b;
        if (b == a.n_seqs - 1) {
            a.rev_tok_off[b + 1] = (b + 1) * a.k;
            a.seq_rev_off[b + 1] = b + 1;
        }
    }
    cluster_wait();
}

// (max, sum of exp) of 16 logits (-inf where there is none) into a running one.
__device__ __forceinline__ void stats16(const float (&x)[16], float& mx, float& z) {
    float cm = mx;
#pragma unroll
    for (int u = 0; u < 16; ++u) cm = fmaxf(cm, x[u]);
    if (cm == -INFINITY) return;
    float cz = 0.0f;
#pragma unroll
    for (int u = 0; u < 16; ++u) cz += __expf(x[u] - cm);
    z = (mx == -INFINITY ? 0.0f : z * __expf(mx - cm)) + cz;
    mx = cm;
}

// Everything after a logits kernel: logits in global memory (mostly L2), read
// once for the statistics and once for the relevances. L2 bounds the large
// ones: 32 sequences x 16,384 tokens x 32 heads (67 MB) on 128 CTAs take ~20
// us: statistics 13k cycles, relevances 11k, the two exchanges 7k, search 6k,
// output 3k. Measured against the three kernels it replaced (normaliser,
// relevance, a top-k of one CTA per sequence counting two bits a round), whole
// selections: that shape 262 -> 244 us, 16 x 8192 cached 72.8 -> 66.9 us, one
// sequence of 16,384 43.9 -> 35.4 us; one of 64 tokens, where the chain of
// exchanges shows, 10.5 -> 14 us of GPU time but 21 -> 16 us with its launches.
constexpr int kTailThreads = 1024;
constexpr int kTailMinTokens = 64;  // per CTA

__global__ void __launch_bounds__(kTailThreads, 1) select_tail_kernel(const __grid_constant__ SelectArgs a) {
    pdl_allow();
    constexpr int NT = kTailThreads, NW = NT / 32;
    __shared__ SelectShared sh;
    extern __shared__ __align__(16) uint32_t keys[];  // [cluster * tok_per_cta] relevances
    const int C = a.cluster, b = int(blockIdx.x) / C, rank = int(cluster_rank());
    const int M = a.n_tokens, Hq = a.n_q_heads;
    const int m_beg = rank * a.tok_per_cta, nt = max(0, min(a.tok_per_cta, M - m_beg));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float* rel = reinterpret_cast<float*>(keys + m_beg);
    const float* lg = a.logits + int64_t(b) * Hq * M + m_beg;
    const bool vec = (M & 3) == 0;  // rows of logits 16-byte aligned (m_beg is a multiple of 16)
    pdl_wait();

    for (int hq = warp; hq < Hq; hq += NW) {
        const float* row = lg + int64_t(hq) * M;
        float mx = -INFINITY, z = 0.0f;
        if (vec) {
            const float4* r4 = reinterpret_cast<const float4*>(row);
            for (int i = lane; i - lane < nt / 4; i += 256) {  // eight 16-byte loads requested together
                float x[2][16];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const float4 v = i + 32 * u < nt / 4 ? r4[i + 32 * u]
                                                         : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
                    float* y = x[u / 4] + 4 * (u % 4);
                    y[0] = v.x; y[1] = v.y; y[2] = v.z; y[3] = v.w;
                }
                stats16(x[0], mx, z);
                stats16(x[1], mx, z);
            }
        } else {
            for (int i = lane; i - lane < nt; i += 512) {
                float x[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) x[u] = i + 32 * u < nt ? row[i + 32 * u] : -INFINITY;
                stats16(x, mx, z);
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const float m2 = __shfl_xor_sync(kAll, mx, o), z2 = __shfl_xor_sync(kAll, z, o);
            merge_max_sum(mx, z, m2, z2);
        }
        if (lane == 0) sh.stat[hq] = make_float2(mx, z);
    }
    merge_stats<NT>(a, C, sh);

    uint32_t lo = 0xffffffffu, hi = 0u;
    auto seen = [&](float r) {
        lo = min(lo, __float_as_uint(r));
        hi = max(hi, __float_as_uint(r));
    };
    if (vec && nt >= 4 * NT) {  // four tokens per thread
        for (int i = tid; i < nt / 4; i += NT) {
            const float4* r4 = reinterpret_cast<const float4*>(lg) + i;
            const int64_t step = M / 4;
            float4 r = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            auto add = [&](const float4& x, int h) {
                const float2 n = sh.norm[h];
                r.x = fmaf(__expf(x.x - n.x), n.y, r.x);
                r.y = fmaf(__expf(x.y - n.x), n.y, r.y);
                r.z = fmaf(__expf(x.z - n.x), n.y, r.z);
                r.w = fmaf(__expf(x.w - n.x), n.y, r.w);
            };
            int h = 0;
            for (; h + 8 <= Hq; h += 8) {  // eight heads' logits requested together
                float4 x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = r4[(h + u) * step];
#pragma unroll
                for (int u = 0; u < 8; ++u) add(x[u], h + u);
            }
            for (; h < Hq; ++h) add(r4[h * step], h);
            reinterpret_cast<float4*>(rel)[i] = r;
            seen(r.x); seen(r.y); seen(r.z); seen(r.w);
            if (a.score_out) {
                float* so = a.score_out + int64_t(b) * M + m_beg + 4 * i;
                so[0] = r.x; so[1] = r.y; so[2] = r.z; so[3] = r.w;
            }
        }
    } else {
        for (int i = tid; i < nt; i += NT) {
            float r = 0.0f;
            int h = 0;
            for (; h + 16 <= Hq; h += 16) {  // sixteen heads' logits requested together
                float x[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) x[u] = lg[int64_t(h + u) * M + i];
#pragma unroll
                for (int u = 0; u < 16; ++u) r = fmaf(__expf(x[u] - sh.norm[h + u].x), sh.norm[h + u].y, r);
            }
            for (; h < Hq; ++h) r = fmaf(__expf(lg[int64_t(h) * M + i] - sh.norm[h].x), sh.norm[h].y, r);
            rel[i] = r;
            seen(r);
            if (a.score_out) a.score_out[int64_t(b) * M + m_beg + i] = r;
        }
    }
    select_topk<NT>(a, b, C, m_beg, nt, keys, lo, hi, sh);
}

cudaLaunchConfig_t cluster_config(int grid, int block, int C, size_t smem, cudaStream_t stream,
                                  cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(grid), 1, 1);
    cfg.blockDim = dim3(unsigned(block), 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(C);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

constexpr size_t kMaxDynSmem = 208 * 1024;  // beside the static shared memory, within 227 KB

// Clusters of 1..16 CTAs of a kernel that the current device holds at once, one
// CTA per SM; found, and the kernel's attributes set, once per device.
using ClusterCounts = std::array<int, kMaxCluster + 1>;
cudaError_t max_clusters(const void* kernel, int block, ClusterCounts* out) {
    static std::mutex mu;
    static std::map<std::pair<int, const void*>, ClusterCounts> cache;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> g(mu);
    const auto key = std::make_pair(dev, kernel);
    auto it = cache.find(key);
    if (it == cache.end()) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kMaxDynSmem));
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        ClusterCounts n{};
        for (int C = 1; C <= kMaxCluster; ++C) {
            cudaLaunchAttribute attr[2];
            cudaLaunchConfig_t cfg = cluster_config(C, block, C, kMaxDynSmem, nullptr, attr);
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&n[size_t(C)], kernel, &cfg) != cudaSuccess) {
                cudaGetLastError();  // a cluster size that this device does not offer
                n[size_t(C)] = 0;
            }
        }
        it = cache.emplace(key, n).first;
    }
    *out = it->second;
    return cudaSuccess;
}

// The largest cluster of which every sequence has one at once, with at least
// min_tok tokens per CTA (but the last); 1 for very large batches.
cudaError_t pick_cluster(const void* kernel, int block, int n_seqs, int n_tokens, int min_tok, int* out) {
    ClusterCounts n;
    const cudaError_t e = max_clusters(kernel, block, &n);
    int C = kMaxCluster;
    while (C > 1 && (n_seqs > n[size_t(C)] || n_tokens <= min_tok * (C - 1))) --C;
    *out = C;
    return e;
}

int tokens_per_cta(int n_tokens, int C) { return ((n_tokens + C - 1) / C + 15) / 16 * 16; }

}  // namespace

cudaError_t launch_select_tail(const SelectArgs& a, int n_seqs, cudaStream_t stream) {
    SelectArgs t = a;
    const void* k = reinterpret_cast<const void*>(select_tail_kernel);
    const cudaError_t e = pick_cluster(k, kTailThreads, n_seqs, a.n_tokens, kTailMinTokens, &t.cluster);
    if (e != cudaSuccess) return e;
    t.tok_per_cta = tokens_per_cta(a.n_tokens, t.cluster);
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config(n_seqs * t.cluster, kTailThreads, t.cluster,
                                                  size_t(t.cluster) * t.tok_per_cta * 4, stream, attr);
    return cudaLaunchKernelEx(&cfg, select_tail_kernel, t);
}
}  // namespace prcr
