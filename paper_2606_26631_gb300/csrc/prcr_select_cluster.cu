// The selection on clusters of CTAs, one cluster per sequence: in one kernel
// from the keys to the indices where the logits fit in the cluster's shared
// memory (select_fused_kernel), else everything after a logits kernel
// (select_tail_kernel), which for cached keys is select_logits_kernel here.
//
// Rank r of a cluster of C CTAs takes the tokens r * T .. r * T + T - 1 of its
// sequence (T = tok_per_cta). Two exchanges through distributed shared memory
// stand where kernel boundaries would:
//   1. softmax statistics: every CTA reduces its tokens' logits to a (max, sum
//      of exp) per query head and writes them into all C CTAs; after a cluster
//      barrier each CTA merges them into the heads' normalisers;
//   2. relevance of the CTA's own tokens (mean over the heads of the softmax
//      weight), written into all of them as well; after a second barrier each
//      CTA holds the whole sequence's relevances.
// (Remote writes before a barrier cost less than remote reads after it.)
// Every CTA then finds the K-th largest relevance by itself (the same answer
// in each) and writes its own tokens' share of the selection in index order,
// knowing from the copy how many lie before its first token. The search
// narrows the range of float bits (relevance >= 0, so bit order is value
// order) that holds the K-th largest: 2048 buckets spread over the range from
// the smallest to the largest relevance, counted by shared-memory atomics
// (about M / 2048 keys meet in a bucket), then the few keys of its bucket
// ranked by one warp; or again over that bucket while it holds many.
#include <algorithm>
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
// `rank` of the cluster, and stores to there.
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(r)
                 : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
    return r;
}
__device__ __forceinline__ void peer_store(uint32_t addr, uint32_t x, uint32_t y) {
    asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(addr), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t addr, const uint4& v) {
    asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

// What the phases share, in static shared memory.
struct SelectShared {
    float2 stat[kSelectMaxQHeads];  // this CTA's (max, sum) per query head
    float2 all[kMaxCluster][kSelectMaxQHeads];  // every CTA's; written by the peers
    float2 norm[kSelectMaxQHeads];  // (max, 1 / (sum * n_q_heads)) over the whole sequence
    uint32_t hist[kBuckets];
    uint2 range[kMaxCluster][32];   // smallest and largest key of every CTA's warps; written by the peers
    uint32_t wsum[32];              // per warp: keys in its buckets; later equal | above << 16 in its tokens
    uint32_t before[2][32];         // per warp: keys equal to X and above it before this CTA's first token
    uint32_t pick[3];               // bucket of the K-th largest, keys in it, keys above it
    uint32_t list[32], n_list;
};

// Exchange 1: the heads' normalisers from every CTA's statistics (stat, visible
// to the CTA), which each CTA writes into all of them. Also sets up the search's
// shared state. The caller has arrived at the cluster barrier once at its start:
// its completion here means that every peer is running.
template <int NT, bool FINE>
__device__ __forceinline__ void merge_stats(const SelectArgs& a, int C, int rank, SelectShared& sh) {
    const int c = threadIdx.x & (kMaxCluster - 1);
    cluster_wait();
    for (int hq = threadIdx.x / kMaxCluster; hq < a.n_q_heads; hq += NT / kMaxCluster) {
        const float2 v = sh.stat[hq];
        if (c < C) peer_store(peer_addr(&sh.all[rank][hq], uint32_t(c)), __float_as_uint(v.x), __float_as_uint(v.y));
    }
    cluster_arrive();
    for (int i = threadIdx.x; i < kBuckets; i += NT) sh.hist[i] = 0u;
    if (threadIdx.x == 0) sh.n_list = 0u;
    cluster_wait();
    for (int h0 = 0; h0 < a.n_q_heads; h0 += NT / kMaxCluster) {
        const int hq = h0 + threadIdx.x / kMaxCluster;
        float2 v = make_float2(-INFINITY, 0.0f);
        if (hq < a.n_q_heads && c < C) v = sh.all[c][hq];
        float m = v.x;
#pragma unroll
        for (int o = kMaxCluster / 2; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kAll, m, o));
        float z = v.y * (v.x == -INFINITY ? 0.0f : exp_term<FINE>(v.x - m));
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
// tokens' relevances at m_beg, which are copied to the peers as theirs are
// here. lo, hi: smallest and largest of the relevances that this thread wrote.
template <int NT>
__device__ __forceinline__ void select_topk(const SelectArgs& a, int b, int C, int m_beg, int nt, uint32_t* keys,
                                            uint32_t lo, uint32_t hi, SelectShared& sh) {
    constexpr int NW = NT / 32, BPT = kBuckets / NT;  // buckets per thread
    const int M = a.n_tokens, T = a.tok_per_cta;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    lo = __reduce_min_sync(kAll, lo);
    hi = __reduce_max_sync(kAll, hi);
    if (lane < C) peer_store(peer_addr(&sh.range[m_beg / T][warp], uint32_t(lane)), lo, hi);
    __syncthreads();  // the CTA's relevances
    {
        const int n4 = (nt + 3) / 4;  // T is a multiple of 16: whole groups of four
        for (int i = tid; i < n4 * C; i += NT) {
            const int c = i / n4, j = m_beg + 4 * (i - c * n4);
            if (c * T != m_beg) peer_store(peer_addr(keys + j, uint32_t(c)), *reinterpret_cast<const uint4*>(keys + j));
        }
    }
    cluster_arrive();
    cluster_wait();
    {
        uint2 v = make_uint2(0xffffffffu, 0u);
        for (int i = lane; i < C * NW; i += 32) {
            const uint2 w = sh.range[i / NW][i % NW];
            v.x = min(v.x, w.x);
            v.y = max(v.y, w.y);
        }
        lo = __reduce_min_sync(kAll, v.x);
        hi = __reduce_max_sync(kAll, v.y);
    }

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
}

// (max, sum of exp) of N logits (-inf where there is none) into a running one. A
// NaN logit makes the sum a NaN, also where no other is finite.
template <bool FINE, int N>
__device__ __forceinline__ void stats_of(const float (&x)[N], float& mx, float& z) {
    float cm = x[0];
#pragma unroll
    for (int u = 1; u < N; ++u) cm = fmaxf(cm, x[u]);
    if (cm == -INFINITY) {  // no logit, unless one is a NaN
#pragma unroll
        for (int u = 0; u < N; ++u) z += x[u] == -INFINITY ? 0.0f : x[u];
        return;
    }
    cm = fmaxf(cm, mx);
    float cz = 0.0f;
#pragma unroll
    for (int u = 0; u < N; ++u) cz += exp_term<FINE>(x[u] - cm);
    z = z * (mx == -INFINITY ? 0.0f : exp_term<FINE>(mx - cm)) + cz;
    mx = cm;
}

// The statistics of a CTA's nt tokens, a warp per query head, from logits in
// global memory.
template <int NW, bool FINE>
__device__ __forceinline__ void tail_stats(const float* lg, int M, int Hq, int nt, bool vec, SelectShared& sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
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
                if (nt <= 128) {  // one load each
                    const float x4[4] = {x[0][0], x[0][1], x[0][2], x[0][3]};
                    stats_of<FINE>(x4, mx, z);
                } else {
                    stats_of<FINE>(x[0], mx, z);
                    stats_of<FINE>(x[1], mx, z);
                }
            }
        } else {
            for (int i = lane; i - lane < nt; i += 512) {
                float x[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) x[u] = i + 32 * u < nt ? row[i + 32 * u] : -INFINITY;
                stats_of<FINE>(x, mx, z);
            }
        }
        float m = mx;
#pragma unroll
        for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kAll, m, o));
        z *= mx == -INFINITY ? 0.0f : exp_term<FINE>(mx - m);
#pragma unroll
        for (int o = 16; o; o >>= 1) z += __shfl_xor_sync(kAll, z, o);
        if (lane == 0) sh.stat[hq] = make_float2(m, z);
    }
}

// Everything after a logits kernel: logits in global memory (mostly L2), read
// once for the statistics and once for the relevances. L2 bounds the large
// ones: 32 sequences x 16,384 tokens x 32 heads (67 MB) on 128 CTAs take ~20
// us: statistics 13k cycles, relevances 11k, the two exchanges 7k, search 6k,
// output 3k. Measured against the three kernels it replaced (normaliser,
// relevance, a top-k of one CTA per sequence counting two bits a round), whole
// selections: that shape 262 -> 243.5 us, one sequence of 16,384 43.9 -> 36 us; one of
// 64 tokens x 4 heads of 112, where the chain of exchanges shows, 19.0 -> 13.6 us in a
// row, as a CUDA graph 12.8 | 12.8.
constexpr int kTailThreads = 1024;
constexpr int kTailMinTokens = 64;  // per CTA

template <bool FINE>
__global__ void __launch_bounds__(kTailThreads, 1) select_tail_kernel(const __grid_constant__ SelectArgs a) {
    constexpr int NT = kTailThreads, NW = NT / 32;
    __shared__ SelectShared sh;
    extern __shared__ __align__(16) uint32_t keys[];  // [cluster * tok_per_cta] relevances
    const int C = a.cluster, b = int(blockIdx.x) / C, rank = int(cluster_rank());
    const int M = a.n_tokens, Hq = a.n_q_heads;
    const int m_beg = rank * a.tok_per_cta, nt = max(0, min(a.tok_per_cta, M - m_beg));
    const int tid = threadIdx.x;
    float* rel = reinterpret_cast<float*>(keys + m_beg);
    const float* lg = a.logits + int64_t(b) * Hq * M + m_beg;
    const bool vec = (M & 3) == 0;  // rows of logits 16-byte aligned (m_beg is a multiple of 16)
    cluster_arrive();
    pdl_wait();

    tail_stats<NW, FINE>(lg, M, Hq, nt, vec, sh);
    __syncthreads();
    // Only now: released at entry, calls in a row pile up (each kernel releases the
    // next before its own wait), and the waiting CTAs of 1024 threads crowd the logits
    // kernel onto few SMs. 8 sequences of 768 tokens x 16 heads of 80 28.0 -> 22.7 us,
    // 1 of 8192 x 16 heads of 256 36.4 -> 29.7, of 112 21.0 -> 20.7; before the search
    // the same.
    pdl_allow();
    merge_stats<NT, FINE>(a, C, rank, sh);
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
                r.x = fmaf(exp_term<FINE>(x.x - n.x), n.y, r.x);
                r.y = fmaf(exp_term<FINE>(x.y - n.x), n.y, r.y);
                r.z = fmaf(exp_term<FINE>(x.z - n.x), n.y, r.z);
                r.w = fmaf(exp_term<FINE>(x.w - n.x), n.y, r.w);
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
                for (int u = 0; u < 16; ++u) r = fmaf(exp_term<FINE>(x[u] - sh.norm[h + u].x), sh.norm[h + u].y, r);
            }
            for (; h < Hq; ++h) r = fmaf(exp_term<FINE>(lg[int64_t(h) * M + i] - sh.norm[h].x), sh.norm[h].y, r);
            rel[i] = r;
            seen(r);
            if (a.score_out) a.score_out[int64_t(b) * M + m_beg + i] = r;
        }
    }
    select_topk<NT>(a, b, C, m_beg, nt, keys, lo, hi, sh);
}

// Shared memory of cta_logits and the fused kernel, in the order of its sections.
struct FusedLayout {
    int pitch;  // floats per head's row of logits: 4 mod 32, free of bank conflicts for the MMA's accumulators
    size_t trig, tok, query, logits, keys, total;
};

__host__ __device__ inline FusedLayout fused_layout(int D, bool cached, int H, int Hq, int T, int C, bool logits = true) {
    FusedLayout f;
    f.pitch = (T + 31) / 32 * 32 + 4;
    f.trig = size_t(H) * D * 32;  // after the queries' fragments [H][D / 16][32] uint4
    const int tiles = T / 16 < 1024 / D ? T / 16 : 1024 / D;
    f.tok = f.trig + (cached ? 0 : size_t(tiles) * D * 64);          // [tiles][D / 8][32] float4
    f.query = f.tok + (size_t(T) * (cached ? 8 : 12) + 15) / 16 * 16;  // rows (int64) or coordinates (3 int32)
    f.logits = f.query + (cached ? size_t(Hq) * (D + 8) * 2 : 0);      // the raw queries
    f.keys = f.logits + (logits ? size_t(Hq) * f.pitch * 4 : 0);
    f.total = f.keys + size_t(C) * T * 4;
    return f;
}

// What depends on the rotary configuration alone, in static shared memory.
template <int D, bool CACHED, int NT>
struct PairTables {
    uint64_t tf[D / 2];                                     // turn rates
    alignas(16) float2 cs[CACHED ? D / 2 : 1];              // (cos, sin) of the query's turn
    uint8_t ax[D / 2];                                      // axes
    __device__ void set(const SelectArgs& a) {
        for (int i = threadIdx.x; i < D / 2; i += NT) {
            tf[i] = a.turn_freq[i];
            ax[i] = uint8_t(pair_axis(i, a.layout, a.sec_t, a.sec_h, a.sec_w));
        }
    }
};

// The NaN logits of a CTA's tokens again, by float32 FMAs: for the rare key or
// query with an infinity, whose remainder is a NaN, where the product with the whole
// operand is an infinity (and a logit of -inf a weight of 0). A call: as code in the
// kernel's path it made a chain with a decode behind it 52.8 -> 55.7 us, though the
// selections alone were as fast.
template <int D, int NT>
__device__ __noinline__ void exact_nans(const SelectArgs& a, int b, int m_beg, int nt, int pitch, float* lg, const uint64_t* tf,
                                        const uint8_t* ax) {
    constexpr int P = D / 2;
    const int64_t p = a.q_pos[b];
    auto value = [](uint16_t w) { return __uint_as_float(uint32_t(w) << 16); };
    for (int e = threadIdx.x; e < a.n_q_heads * nt; e += NT) {
        const int hq = e / nt, t = e - hq * nt;
        if (lg[hq * pitch + t] == lg[hq * pitch + t]) continue;
        const uint16_t* q = a.q + (int64_t(b) * a.n_q_heads + hq) * D;
        const uint16_t* k = a.store_k + int64_t(b) * a.store_seq_stride + int64_t(a.layer) * a.store_layer_stride +
                            int64_t(m_beg + t) * a.store_token_stride + int64_t(hq / (a.n_q_heads / a.n_kv_heads)) * D;
        const int32_t* crd = a.coords + int64_t(b) * a.coord_seq_stride + 3 * int64_t(m_beg + t);
        float sum = 0.0f;
        for (int i = 0; i < P; ++i) {
            float sn, cs;
            sincos_coord(int64_t(crd[ax[i]]) - p, tf[i], &sn, &cs);
            const float x = value(k[i]), y = value(k[i + P]);
            sum = fmaf(value(q[i]), fmaf(x, cs, -y * sn), sum);
            sum = fmaf(value(q[i + P]), fmaf(y, cs, x * sn), sum);
        }
        lg[hq * pitch + t] = sum * a.scale;
    }
    __syncthreads();
}

// Logits of tokens m_beg .. m_beg + nt - 1 of sequence b for the query heads of
// KV heads kh0 .. kh0 + H - 1: query head kh0 g + h, token m_beg + t at
// lg[h * lg_pitch + t]. Raw keys are turned by the offsets of their
// coordinates as in ads_logits_mma_kernel (CACHED = false); position-bound rows
// meet the query turned at (p, p, p), a bf16 head and remainder (CACHED = true;
// the bf16 keys are exact operands, S^T = K Q^T by m16n8k16). A work item is
// (16 tokens, KV head), and the CTA's warps take them in turn, heads fastest;
// an item's rows are loaded during the item before. The queries' fragments,
// the cache rows of the tokens, and the raw keys' cos/sin (a pass of 1024 / D
// tiles at a time) are found once per CTA.
template <int D, bool CACHED, int NT>
__device__ __forceinline__ void cta_logits(const SelectArgs& a, const FusedLayout& f, int b, int kh0, int H, int m_beg,
                                           int nt, unsigned char* smem_raw, PairTables<D, CACHED, NT>& pt, float* lg,
                                           int lg_pitch, uint32_t& err) {
    constexpr int NW = NT / 32, P = D / 2;
    constexpr int KQ = D / 16;                  // 16-byte fragment entries per lane of a KV head's queries
    constexpr int NR = CACHED ? D / 32 : D / 64;  // groups of 16-byte loads of an item, refilled as they are used
    constexpr int RL = CACHED ? 2 : 4;            // loads per group
    constexpr int TP = 1024 / D;                // tiles of a pass (raw keys)
    constexpr int QP = D + 8;                   // bf16 per staged query row
    const int Hq = a.n_q_heads, g = Hq / a.n_kv_heads, n_tiles = (nt + 15) / 16;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tq = lane & 3;
    uint4* qf_s = reinterpret_cast<uint4*>(smem_raw);
    float4* tr_s = reinterpret_cast<float4*>(smem_raw + f.trig);
    int* crd_s = reinterpret_cast<int*>(smem_raw + f.tok);
    int64_t* row_s = reinterpret_cast<int64_t*>(smem_raw + f.tok);
    uint32_t* q_s = reinterpret_cast<uint32_t*>(smem_raw + f.query);
    const int64_t p = a.q_pos[b];
    const uint16_t* qs = a.q + (int64_t(b) * Hq + kh0 * g) * D;

    // the items of this warp: warp, warp + NW, ... of (tile, KV head), heads fastest
    uint4 k[NR][RL];
    const uint16_t* kb = CACHED ? a.cache_k + int64_t(a.layer) * a.cache_layer_stride + kh0 * a.cache_head_stride + 8 * tq
                                : a.store_k + int64_t(b) * a.store_seq_stride + int64_t(m_beg) * a.store_token_stride +
                                      int64_t(a.layer) * a.store_layer_stride + kh0 * D + 8 * tq;
    // this lane's two token rows (gid and gid + 8 of the tile) at KV head kh; a
    // token past the end reads the last one, one without a row the cache's
    // first row (their logits are not stored, or are -inf)
    auto rows = [&](int tile, int kh, const uint16_t* (&r)[2]) {
        const int ta = min(16 * tile + gid, nt - 1), tb = min(16 * tile + gid + 8, nt - 1);
        if constexpr (CACHED) {
            const int64_t ra = row_s[ta], rb = row_s[tb];
            r[0] = kb + (ra < 0 ? 0 : ra) + kh * a.cache_head_stride;
            r[1] = kb + (rb < 0 ? 0 : rb) + kh * a.cache_head_stride;
        } else {
            r[0] = kb + int64_t(ta) * a.store_token_stride + kh * D;
            r[1] = kb + int64_t(tb) * a.store_token_stride + kh * D;
        }
    };
    auto fetch = [&](uint4 (&x)[RL], const uint16_t* ra, const uint16_t* rb, int u) {
        if constexpr (CACHED) {
            x[0] = ld_stream(ra + 32 * u);
            x[1] = ld_stream(rb + 32 * u);
        } else {
            x[0] = ld_stream(ra + 32 * u);
            x[1] = ld_stream(ra + 32 * u + P);
            x[2] = ld_stream(rb + 32 * u);
            x[3] = ld_stream(rb + 32 * u + P);
        }
    };
    const int n_items = n_tiles * H;
    const uint16_t* r_n[2];
    auto first = [&]() {
        if (warp < n_items) {
            rows(warp / H, warp % H, r_n);
#pragma unroll
            for (int u = 0; u < NR; ++u) fetch(k[u], r_n[0], r_n[1], u);
        }
    };
    const uint32_t* q_src = reinterpret_cast<const uint32_t*>(qs);  // 4-byte loads: the ABI's alignment
    // B fragments of the groups' query heads: one entry per (KV head, j, head of
    // the group, lane group t); those past the group's heads stay zero
    auto each_fragment = [&](auto&& make) {
        if (g < 8)
            for (int e = tid; e < H * KQ * 32; e += NT)
                if (gid >= g) qf_s[e] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 4
        for (int e = tid; e < H * KQ * g * 4; e += NT) {
            const int t = e & 3, h = (e >> 2) % g, kj = (e >> 2) / g;
            const int kh = kj / KQ, j = kj % KQ;
            qf_s[kj * 32 + 4 * h + t] = make(kh * g + h, j, t);
        }
    };
    bool q_ok = true;
    if constexpr (CACHED) {
        // the query rows into shared memory, the cache rows of the CTA's tokens
        // (-1: none), and the query's turn
#pragma unroll 4
        for (int i = tid; i < H * g * P; i += NT) q_s[(i / P) * (QP / 2) + i % P] = __ldg(q_src + i);
        const int64_t s0 = a.img_slot0[b];
        for (int t = tid; t < nt; t += NT) {
            const int64_t slot = s0 + m_beg + t;
            int64_t row = -1;
            if (slot < 0 || slot >= a.cache_capacity) {
                err |= PRCR_ST_CAPACITY;
            } else if (a.cache_kind == PRCR_CACHE_CONTIGUOUS) {
                row = int64_t(b) * a.cache_seq_stride + slot * a.cache_slot_stride;
            } else {
                const int64_t lb = slot <= INT32_MAX ? int64_t(uint32_t(slot) / uint32_t(a.block_size))
                                                     : slot / a.block_size;
                const int32_t blk = a.block_table[int64_t(b) * a.bt_stride + lb];
                if (blk < 0 || blk >= a.n_blocks) err |= PRCR_ST_NO_BLOCK;
                else row = int64_t(blk) * a.cache_block_stride + (slot - lb * a.block_size) * a.cache_slot_stride;
            }
            row_s[t] = row;
        }
        // a query position beyond the fixed-point angle reduction is reported
        // and the sequence's logits are all -inf (relevance 0)
        q_ok = p > -2147483648LL && p < 2147483648LL;
        if (!q_ok) err |= PRCR_ST_POS_RANGE;
        for (int i = tid; i < P; i += NT) {
            float sn, cs;
            sincos_fixed(q_ok ? static_cast<long long>(p) * (1ll << 32) : 0ll, pt.tf[i], &sn, &cs);
            pt.cs[i] = make_float2(cs, sn);
        }
        __syncthreads();
        first();
        // four dimensions of 16-byte chunk t + 4 (j / 2) (the chunks that the
        // lane loads of its keys: the four lanes of a token cover 64 contiguous
        // bytes per load), turned at (p, p, p) and scaled, a bf16 head and
        // remainder each
        each_fragment([&](int hq, int j, int t) {
            const uint32_t* q0 = q_s + hq * (QP / 2);
            const int d = 8 * (t + 4 * (j >> 1)) + 4 * (j & 1), dp = d < P ? d + P : d - P, i = d < P ? d : dp;
            const uint2 x = *reinterpret_cast<const uint2*>(q0 + d / 2), y = *reinterpret_cast<const uint2*>(q0 + dp / 2);
            const float4 ca = *reinterpret_cast<const float4*>(pt.cs + i), cb = *reinterpret_cast<const float4*>(pt.cs + i + 2);
            const float sg = d < P ? -1.0f : 1.0f;
            uint4 o;
            split_bf16x2(fmaf(lo_f32(x.x), ca.x, sg * lo_f32(y.x) * ca.y) * a.scale,
                         fmaf(hi_f32(x.x), ca.z, sg * hi_f32(y.x) * ca.w) * a.scale, o.x, o.z);
            split_bf16x2(fmaf(lo_f32(x.y), cb.x, sg * lo_f32(y.y) * cb.y) * a.scale,
                         fmaf(hi_f32(x.y), cb.z, sg * hi_f32(y.y) * cb.w) * a.scale, o.y, o.w);
            return o;
        });
        __syncthreads();
    } else {
        first();
        const int32_t* crd = a.coords + int64_t(b) * a.coord_seq_stride + 3 * int64_t(m_beg);
        for (int i = tid; i < 3 * nt; i += NT) crd_s[i] = crd[i];
        // the raw query at k-steps 2j and 2j + 1 (exact tf32 operands), whose
        // pairs are neighbours: one word of each half
        each_fragment([&](int hq, int j, int t) {
            const uint32_t* q0 = q_src + hq * P + 16 * (j / 4) + 4 * t + j % 4;
            const uint32_t w0 = __ldg(q0), w1 = __ldg(q0 + P / 2);
            return make_uint4(w0 << 16, w1 << 16, w0 & 0xffff0000u, w1 & 0xffff0000u);
        });
        __syncthreads();
    }

    constexpr int STEP = CACHED ? 1 << 28 : TP;  // tiles per pass
    for (int t0 = 0, it = warp; t0 < n_tiles; t0 += STEP) {
        const int t1 = min(n_tiles, t0 + STEP);
        if constexpr (!CACHED) {
            // cos/sin of (token, pair) at each k-step, in the lanes' order
            if (t0) __syncthreads();  // the previous pass has been read
            for (int e = tid; e < (t1 - t0) * (D / 8) * 32; e += NT) {
                const int s = (e / 32) % (D / 8), tile = t0 + e / (32 * (D / 8));
                const int i = 32 * (s / 8) + 8 * tq + s % 8, ax = pt.ax[i];
                const int ta = min(16 * tile + gid, nt - 1), tb = min(16 * tile + gid + 8, nt - 1);
                float4 v;
                sincos_coord(int64_t(crd_s[3 * ta + ax]) - p, pt.tf[i], &v.z, &v.x);
                sincos_coord(int64_t(crd_s[3 * tb + ax]) - p, pt.tf[i], &v.w, &v.y);
                tr_s[e] = v;
            }
            __syncthreads();
        }
        for (; it < t1 * H; it += NW) {
            const int tile = it / H, kh = it - tile * H;
            const bool more = it + NW < n_items;
            if (more) rows((it + NW) / H, (it + NW) % H, r_n);
            constexpr int NC = CACHED ? 4 : 2;  // accumulator chains per head
            float acc[NC][4], lead[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int u = 0; u < NC; ++u) acc[u][0] = acc[u][1] = acc[u][2] = acc[u][3] = 0.0f;
            const uint4* qf = qf_s + kh * KQ * 32 + lane;
            if constexpr (CACHED) {
#pragma unroll
                for (int u = 0; u < NR; ++u) {
                    const uint4 w0 = k[u][0], w1 = k[u][1];
                    const uint4 qa = qf[(2 * u) * 32], qb = qf[(2 * u + 1) * 32];
                    mma_16816(acc[0], w0.x, w1.x, w0.y, w1.y, qa.x, qa.y);
                    mma_16816(acc[1], w0.x, w1.x, w0.y, w1.y, qa.z, qa.w);
                    mma_16816(acc[NC - 2], w0.z, w1.z, w0.w, w1.w, qb.x, qb.y);
                    mma_16816(acc[NC - 1], w0.z, w1.z, w0.w, w1.w, qb.z, qb.w);
                    if (more) fetch(k[u], r_n[0], r_n[1], u);
                }
            } else {
                const float4* tr = tr_s + (tile - t0) * (D / 8) * 32 + lane;
#pragma unroll
                for (int u = 0; u < NR; ++u) {
#pragma unroll
                    for (int s8 = 0; s8 < 8; ++s8) {
                        const int w = s8 / 2;
                        const bool up = s8 & 1;  // upper bf16 of the word
                        const float4 t = tr[(8 * u + s8) * 32];
                        const float2 Cs = make_float2(t.x, t.y), Sn = make_float2(t.z, t.w);
                        const uint32_t xa = word_of(k[u][0], w), ya = word_of(k[u][1], w);
                        const uint32_t xb = word_of(k[u][2], w), yb = word_of(k[u][3], w);
                        const float2 X = up ? make_float2(hi_f32(xa), hi_f32(xb)) : make_float2(lo_f32(xa), lo_f32(xb));
                        const float2 Y = up ? make_float2(hi_f32(ya), hi_f32(yb)) : make_float2(lo_f32(ya), lo_f32(yb));
                        const float2 ys = __fmul2_rn(Y, Sn), xs = __fmul2_rn(X, Sn);
                        const float2 Xr = __ffma2_rn(X, Cs, make_float2(-ys.x, -ys.y));
                        const float2 Yr = __ffma2_rn(Y, Cs, xs);
                        // tf32 heads by truncation, float32 remainders
                        const uint32_t hxa = __float_as_uint(Xr.x) & 0xffffe000u, hxb = __float_as_uint(Xr.y) & 0xffffe000u;
                        const uint32_t hya = __float_as_uint(Yr.x) & 0xffffe000u, hyb = __float_as_uint(Yr.y) & 0xffffe000u;
                        const float2 lx = __ffma2_rn(make_float2(__uint_as_float(hxa), __uint_as_float(hxb)),
                                                     make_float2(-1.0f, -1.0f), Xr);
                        const float2 ly = __ffma2_rn(make_float2(__uint_as_float(hya), __uint_as_float(hyb)),
                                                     make_float2(-1.0f, -1.0f), Yr);
                        const uint4 q2 = qf[(4 * u + w) * 32];
                        const uint32_t b0 = up ? q2.z : q2.x, b1 = up ? q2.w : q2.y;
                        // head_dim 256: remainders rounded (half a tf32 unit added) and, the
                        // tensor core truncating what it adds, the leading chain cut every
                        // two k-steps and added with its rounding error kept (Knuth's
                        // two-sum). Error against float64 0.8e-7 to 1.5e-7, of one chain 2.7e-7
                        // to 7e-7 (float32 FMAs on the CUDA cores 1.1e-7 to 1.7e-7); 13
                        // sequences of 456 tokens x 8 heads 15.9 -> 17.4 us (CUDA cores 48.8).
                        constexpr uint32_t kHalf = D == 256 ? 0x1000u : 0u;
                        mma_1688_tf32(acc[0], hxa, hxb, hya, hyb, b0, b1);
                        mma_1688_tf32(acc[1], __float_as_uint(lx.x) + kHalf, __float_as_uint(lx.y) + kHalf, __float_as_uint(ly.x) + kHalf,
                                      __float_as_uint(ly.y) + kHalf, b0, b1);
                        if (D == 256 && s8 % 2 == 1) {
#pragma unroll
                            for (int v = 0; v < 4; ++v) {
                                const float sum = lead[v] + acc[0][v], part = sum - lead[v];
                                acc[1][v] += (lead[v] - (sum - part)) + (acc[0][v] - part);
                                lead[v] = sum;
                                acc[0][v] = 0.0f;
                            }
                        }
                    }
                    if (more) fetch(k[u], r_n[0], r_n[1], u);
                }
            }
            // rows gid and gid + 8 (tokens), columns 2 tq and 2 tq + 1 (heads of the group)
            const int ta = 16 * tile + gid, tb = ta + 8;
            bool ok_a = true, ok_b = true;
            if constexpr (CACHED) {
                ok_a = q_ok && row_s[min(ta, nt - 1)] >= 0;
                ok_b = q_ok && row_s[min(tb, nt - 1)] >= 0;
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (2 * tq + c >= g) continue;
                float va, vb;
                if constexpr (CACHED) {  // chains 1 and 3: the query's remainder
                    va = (acc[1][c] + acc[NC - 1][c]) + (acc[0][c] + acc[NC - 2][c]);
                    vb = (acc[1][2 + c] + acc[NC - 1][2 + c]) + (acc[0][2 + c] + acc[NC - 2][2 + c]);
                } else {  // chain 1: the keys' remainders (and lead's rounding errors)
                    va = ((D == 256 ? lead[c] : acc[0][c]) + acc[1][c]) * a.scale;
                    vb = ((D == 256 ? lead[2 + c] : acc[0][2 + c]) + acc[1][2 + c]) * a.scale;
                }
                float* dst = lg + (kh * g + 2 * tq + c) * lg_pitch;
                if (ta < nt) dst[ta] = ok_a ? va : -INFINITY;
                if (tb < nt) dst[tb] = ok_b ? vb : -INFINITY;
            }
        }
    }
}

// (max, sum of exp) per query head of nt tokens' logits in shared memory, two
// heads of a warp side by side. True where one of this thread's sums is a NaN.
template <int NT>
__device__ __forceinline__ bool cta_stats(const float* lg_s, int pitch, int Hq, int nt, float2* stat) {
    bool nan = false;
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int h0 = warp; h0 < Hq; h0 += 2 * NW) {
        const bool two = h0 + NW < Hq;
        const float* ra = lg_s + h0 * pitch;
        const float* rb = lg_s + (two ? h0 + NW : h0) * pitch;
        float ma = -INFINITY, mb = -INFINITY, za = 0.0f, zb = 0.0f;
        for (int t = lane; t < nt; t += 32) {
            ma = fmaxf(ma, ra[t]);
            mb = fmaxf(mb, rb[t]);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            ma = fmaxf(ma, __shfl_xor_sync(kAll, ma, o));
            mb = fmaxf(mb, __shfl_xor_sync(kAll, mb, o));
        }
        const float sa = ma == -INFINITY ? 0.0f : ma, sb = mb == -INFINITY ? 0.0f : mb;
        for (int t = lane; t < nt; t += 32) {
            za += __expf(ra[t] - sa);
            zb += __expf(rb[t] - sb);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            za += __shfl_xor_sync(kAll, za, o);
            zb += __shfl_xor_sync(kAll, zb, o);
        }
        if (lane == 0) {
            stat[h0] = make_float2(ma, za);
            if (two) stat[h0 + NW] = make_float2(mb, zb);
        }
        nan = nan || za != za || zb != zb;
    }
    return nan;
}

// The whole selection in one kernel; the CTA's logits stay in shared memory.
// Small calls are a chain of latencies, which one kernel shortens by three
// launches: 768 tokens x 8 KV heads in a cluster of 16, ~20k cycles: queries
// and first rows 2.7k, cos/sin and MMAs 5.5k, statistics and their exchange
// 4.8k, relevances and theirs 5k, search and output 2.7k. Measured with its
// launches 20.9 -> 11.5 us (four kernels before), 8 sequences 20.1 -> 13.1 us,
// 4 of 1000 tokens at head_dim 256 29.7 -> 14.7 us (CUDA cores before).
constexpr int kFusedThreads = 512;

template <int D, bool CACHED>
__global__ void __launch_bounds__(kFusedThreads, 1) select_fused_kernel(const __grid_constant__ SelectArgs a) {
    constexpr int NT = kFusedThreads;
    __shared__ SelectShared sh;
    __shared__ PairTables<D, CACHED, NT> pt;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_allow();
    const int C = a.cluster, b = int(blockIdx.x) / C, rank = int(cluster_rank()), T = a.tok_per_cta;
    const int M = a.n_tokens, Hq = a.n_q_heads;
    const int m_beg = rank * T, nt = max(0, min(T, M - m_beg));
    const int tid = threadIdx.x;
    const FusedLayout f = fused_layout(D, CACHED, a.n_kv_heads, Hq, T, C);
    float* lg_s = reinterpret_cast<float*>(smem_raw + f.logits);
    uint32_t* keys = reinterpret_cast<uint32_t*>(smem_raw + f.keys);
    pt.set(a);
    cluster_arrive();
    uint32_t err = 0;
    pdl_wait();
    cta_logits<D, CACHED, NT>(a, f, b, 0, a.n_kv_heads, m_beg, nt, smem_raw, pt, lg_s, f.pitch, err);
    if (CACHED && err) atomicOr(a.status, err);
    __syncthreads();
    if constexpr (D == 256 && !CACHED) {
        for (bool again = true; __syncthreads_or(cta_stats<NT>(lg_s, f.pitch, Hq, nt, sh.stat)) && again; again = false)
            exact_nans<D, NT>(a, b, m_beg, nt, f.pitch, lg_s, pt.tf, pt.ax);
    } else {
        cta_stats<NT>(lg_s, f.pitch, Hq, nt, sh.stat);
        __syncthreads();
    }
    merge_stats<NT, false>(a, C, rank, sh);

    // relevances: `per` lanes share a token (its heads in turn) where the CTA
    // has few tokens
    float* rel = reinterpret_cast<float*>(keys + m_beg);
    const int per = nt * 8 <= NT ? 8 : (nt * 4 <= NT ? 4 : (nt * 2 <= NT ? 2 : 1));
    uint32_t lo = 0xffffffffu, hi = 0u;
    for (int i0 = 0; i0 < nt * per; i0 += NT) {
        const int t = (i0 + tid) / per, j = (i0 + tid) & (per - 1);
        float r = 0.0f;
        if (t < nt)
            for (int h = j; h < Hq; h += per) r = fmaf(__expf(lg_s[h * f.pitch + t] - sh.norm[h].x), sh.norm[h].y, r);
        for (int o = per / 2; o; o >>= 1) r += __shfl_xor_sync(kAll, r, o);
        if (t < nt && j == 0) {
            rel[t] = r;
            lo = min(lo, __float_as_uint(r));
            hi = max(hi, __float_as_uint(r));
            if (a.score_out) a.score_out[int64_t(b) * M + m_beg + t] = r;
        }
    }
    select_topk<NT>(a, b, C, m_beg, nt, keys, lo, hi, sh);
}

// Logits of the cached-key selection to global memory, where it is too large for
// one cluster per sequence: a CTA takes one (sequence, chunk of tok_per_cta
// tokens, group of kh_per_item KV heads), two CTAs per SM (four at head_dim 64,
// whose items are half as long), so that one's set-up runs beside the other's
// streaming. DRAM bounds it, with 64 KB of keys in flight per SM; these need lines of L1, so shared memory is kept small (logits staged
// there for whole-line stores and statistics, 200 KB per SM, made it 2 to 3
// times slower). Measured against a kernel whose warps each looked up their rows
// per item and loaded 64 bytes per lane (half a sector per load), whole selections:
// 16 sequences of 8192 tokens x 8 heads of 128 66.8 -> 63.1 us, 32 of 16,384 212.6
// -> 206.0 us, 16 of 4096 40.1 -> 36.6 us, 7 of 8192 40.3 -> 36.0 us. Head_dim
// 64, 32 sequences of 8192 x 8 heads, before | two | three | four | five CTAs per SM:
// 71.9 | 76.3 | 61.6 | 59.8 | 73.6.
constexpr int kSplitThreads = 256;
template <int D>
constexpr int kSplitCtas = D == 64 ? 4 : 2;  // per SM

template <int D>
__global__ void __launch_bounds__(kSplitThreads, kSplitCtas<D>) select_logits_kernel(const __grid_constant__ SelectArgs a) {
    constexpr int NT = kSplitThreads;
    __shared__ PairTables<D, true, NT> pt;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Hq = a.n_q_heads, H = a.n_kv_heads, g = Hq / H, M = a.n_tokens, T = a.tok_per_cta;
    const int n_hg = (H + a.kh_per_item - 1) / a.kh_per_item, n_chunks = (M + T - 1) / T;
    const int unit = int(blockIdx.x) / n_hg, kh0 = (int(blockIdx.x) - unit * n_hg) * a.kh_per_item;
    const int b = unit / n_chunks, m_beg = (unit - b * n_chunks) * T;
    const FusedLayout f = fused_layout(D, true, a.kh_per_item, a.kh_per_item * g, T, 0, false);
    pdl_allow();
    pt.set(a);
    uint32_t err = 0;
    pdl_wait();
    cta_logits<D, true, NT>(a, f, b, kh0, min(a.kh_per_item, H - kh0), m_beg, min(T, M - m_beg), smem_raw, pt,
                            a.logits + (int64_t(b) * Hq + kh0 * g) * M + m_beg, M, err);
    if (err) atomicOr(a.status, err);
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

constexpr int kFusedMinTokens = 32;  // per CTA
constexpr int kSplitMinTokens = 64, kSplitMaxTokens = 2048;  // per CTA of the logits kernel
constexpr size_t kMaxDynSmem = 192 * 1024;  // beside the static shared memory, within 227 KB

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

cudaError_t launch_select_tail(const SelectArgs& a, int n_seqs, bool fine, cudaStream_t stream) {
    SelectArgs t = a;
    auto kern = fine ? select_tail_kernel<true> : select_tail_kernel<false>;
    const void* k = reinterpret_cast<const void*>(kern);
    const cudaError_t e = pick_cluster(k, kTailThreads, n_seqs, a.n_tokens, kTailMinTokens, &t.cluster);
    if (e != cudaSuccess) return e;
    t.tok_per_cta = tokens_per_cta(a.n_tokens, t.cluster);
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config(n_seqs * t.cluster, kTailThreads, t.cluster,
                                                  size_t(t.cluster) * t.tok_per_cta * 4, stream, attr);
    return cudaLaunchKernelEx(&cfg, kern, t);
}

// The one-kernel selection, or *done = false where it does not fit or is the
// slower path. It leaves SMs idle (a cluster per sequence, and clusters do not
// fill every GPC), so its time grows with the work of a CTA, that of a logits
// kernel and select_tail_kernel with all work over all SMs, on top of a few us more
// for the second kernel. Work is counted in key rows (token, KV head), to which raw
// keys add about three per token for its cos/sin; the second path grows with their
// number per SM, at first faster (its grids fill) than in proportion. The constants are
// fitted per head_dim to 41,871 drawn calls timed both ways (1..48 sequences of
// 128..16,384 tokens, 1..8 KV heads, groups of 1..7) and 7080 of 9..64 KV heads: the
// chosen path is 0.1 to 0.4 % behind the better one on average, with more heads 0.5 to
// 1 % (3.6 % cached at 256); with one line for all head dims, linear, in rows of 128,
// 0.6 to 2.6 %, 1.3 to 13 %, and twice as slow at worst. Some of them, us, fused | two kernels: raw
// keys, 8 heads of 128, 1 sequence of 1024 tokens 12.2 | 12.9, of 1536 14.2 | 13.3; 7 of
// 4096 27.5 | 30.2; 40 of 2048 x 8 heads of 64 46.0 | 36.2, 7 of 8192 37.1 | 29.9; 1 of
// 1024 x 8 of 256 18.0 | 26.3. Cached keys, 8 heads of 128, 1 of 2048 13.3 | 13.7, of
// 3072 15.8 | 14.7; 7 of 4096 18.8 | 19.8; 16 of 4096 43 | 35; 8 heads of 256, 7 of 1536
// 16.6 | 17.2, of 3072 24.4 | 22.9.
struct FusedLine {
    double rows, heads, linear, root;
};
constexpr FusedLine kFusedLine[2][3] = {{{590, 10, 0.33, 52}, {330, 0, 0.2, 55}, {490, 7, 1.5, 27}},   // raw keys: head_dim 64, 128, 256
                                        {{850, 37, 0.16, 30}, {600, 5, 0.75, 9}, {280, 0, 0.7, 17}}};  // cached keys
template <int D, bool CACHED>
cudaError_t try_fused(const SelectArgs& a, int n_seqs, int sms, cudaStream_t stream, bool* done) {
    auto kern = select_fused_kernel<D, CACHED>;
    const void* k = reinterpret_cast<const void*>(kern);
    SelectArgs t = a;
    cudaError_t e = pick_cluster(k, kFusedThreads, n_seqs, a.n_tokens, kFusedMinTokens, &t.cluster);
    if (e != cudaSuccess) return e;
    t.tok_per_cta = tokens_per_cta(a.n_tokens, t.cluster);
    const FusedLayout f = fused_layout(D, CACHED, a.n_kv_heads, a.n_q_heads, t.tok_per_cta, t.cluster);
    const int64_t per_token = a.n_kv_heads + (CACHED ? 0 : 3);
    const double spread = double(n_seqs) * a.n_tokens * per_token / sms;
    const FusedLine c = kFusedLine[CACHED][D / 128];
    const double line = c.rows + c.heads * per_token + c.linear * spread + c.root * std::sqrt(spread);
    if (f.total > kMaxDynSmem || double(t.tok_per_cta * per_token) > line) return cudaSuccess;
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config(n_seqs * t.cluster, kFusedThreads, t.cluster, f.total, stream, attr);
    *done = true;
    return cudaLaunchKernelEx(&cfg, kern, t);
}

// Chunks of the cached-key logits: as many per sequence as make one wave of
// kSplitCtas CTAs per SM, of at least kSplitMinTokens tokens and at most kSplitMaxTokens.
template <int D>
cudaError_t launch_logits_split(const SelectArgs& a, int n_seqs, int sms, cudaStream_t stream) {
    SelectArgs t = a;
    const int H = a.n_kv_heads, g = a.n_q_heads / H;
    t.kh_per_item = H < 1024 / D ? H : 1024 / D;  // 32 KB of query fragments at most
    const int64_t per = int64_t(n_seqs) * ((H + t.kh_per_item - 1) / t.kh_per_item);
    const int64_t n = std::max<int64_t>(1, kSplitCtas<D> * int64_t(sms) / per);
    const int64_t T = std::min<int64_t>(kSplitMaxTokens, std::max<int64_t>(kSplitMinTokens, (a.n_tokens + n - 1) / n));
    t.tok_per_cta = int((T + 15) / 16 * 16);
    const size_t smem = fused_layout(D, true, t.kh_per_item, t.kh_per_item * g, t.tok_per_cta, 0, false).total;
    const int64_t grid = per * ((a.n_tokens + t.tok_per_cta - 1) / t.tok_per_cta);
    if (grid > INT32_MAX) return cudaErrorInvalidValue;
    const cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(select_logits_kernel<D>), smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(select_logits_kernel<D>, dim3(unsigned(grid)), dim3(kSplitThreads), smem, stream, t);
}

cudaError_t launch_select_cached_logits(const SelectArgs& a, int n_seqs, int sms, cudaStream_t stream) {
    return a.head_dim == 64    ? launch_logits_split<64>(a, n_seqs, sms, stream)
           : a.head_dim == 128 ? launch_logits_split<128>(a, n_seqs, sms, stream)
                               : launch_logits_split<256>(a, n_seqs, sms, stream);
}

cudaError_t launch_select_fused(const SelectArgs& a, bool cached, int n_seqs, int sms, cudaStream_t stream, bool* done) {
    *done = false;
    if (a.head_dim == 64) return cached ? try_fused<64, true>(a, n_seqs, sms, stream, done) : try_fused<64, false>(a, n_seqs, sms, stream, done);
    if (a.head_dim == 128) return cached ? try_fused<128, true>(a, n_seqs, sms, stream, done) : try_fused<128, false>(a, n_seqs, sms, stream, done);
    if (a.head_dim == 256) return cached ? try_fused<256, true>(a, n_seqs, sms, stream, done) : try_fused<256, false>(a, n_seqs, sms, stream, done);
    return cudaSuccess;
}
}  // namespace prcr
