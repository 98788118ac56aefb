// Attention-driven selection of the revisited set (Sec. 2.1, Eq. 3).
//
// The paper names the selection module and what it does (rank the visual
// tokens by relevance to the current decoding context, keep K of them) but
// not its formula. Reading implemented here: relevance of visual token m is
// the trigger query's attention on m at one layer, a softmax over the M
// visual tokens of RoPE(q_h, (p, p, p)) . RoPE(k_m, p_m) / sqrt(D) per query
// head h (GQA: head h reads KV head h / group), averaged over the heads. The
// K most relevant tokens (equal relevance: lower token index first) are
// written in ascending token order, one revisit per sequence, as the offsets
// and indices prcr_rebind_inject takes.
//
// A rotation preserves dot products and composes by adding angles, so
// RoPE(q, (p, p, p)) . RoPE(k, c) = q . R(c - p) k: pair i of the raw key is
// turned by theta_i (c_axis(i) - p) and dotted with the raw query, and the
// 1/sqrt(D) scale is applied to the dot product. The raw bf16 query is then
// exact in any operand format, and nothing is computed per query.
// The logits kernels here (from the raw keys, rotated on the fly) write every
// (token, query head) logit to the workspace; prcr_select_cluster.cu does the
// rest: softmax normalisers, relevances, top-k; and all of it for small calls
// and for the keys of the position-bound cache.
#include <cmath>

#include "prcr_pdl.cuh"
#include "prcr_select.cuh"

namespace prcr {
namespace {

// 16-byte chunk c of a shared row stored at c ^ bit 3 of c: the 8 lanes of a
// quarter-warp that read chunks 2v (or 2v + 1), v = 0..7, hit 8 distinct
// bank groups.
__device__ __forceinline__ int swz(int c) { return c ^ ((c >> 3) & 1); }

// Logits of every (token, query head). Persistent: CTA c takes a contiguous
// run of the B * n_tiles token tiles (sequence-major), so it reloads the
// rotated queries only when its run enters a new sequence. Per tile of T
// tokens: the tile's cos/sin (one per token and pair) go to shared memory;
// then each row (token, KV head) is taken by L lanes, lane v holding pairs
// 8v..8v+7 (one 16-byte load from each half of the raw key row), which it
// rotates and dots with the group's query heads in packed float2 FMAs; the
// lanes' partial sums are reduced by shuffles. The loads of a lane's next two
// rows are in flight during the current row's arithmetic. The tile's logits are staged
// in shared memory and written out coalesced.
// L lanes per row (a power of two >= head_dim / 16); G = the GQA group size g
// for g = 1, 2 and 4, else 8 (heads h >= g skipped).
template <int L, int G>
__global__ void __launch_bounds__(256, 3) ads_logits_kernel(const __grid_constant__ SelectArgs a) {
    pdl_allow();
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    const int D = a.head_dim, P = D >> 1, Hq = a.n_q_heads, H = a.n_kv_heads, g = Hq / H;
    const int NV = P >> 3, M = a.n_tokens, T = a.tok_tile;
    const int qrow = D / 4 + 1;  // chunks per row; odd, so adjacent rows fall in other banks
    const int crow = P / 4 + 1;
    float4* q_s = reinterpret_cast<float4*>(sm);  // row h * H + kh holds query head kh * g + h
    float4* c_s = q_s + Hq * qrow;                // [T] cos rows
    float4* s_s = c_s + T * crow;                 // [T] sin rows
    float* lg_s = reinterpret_cast<float*>(s_s + T * crow);  // [Hq][T + 1]
    int* crd_s = reinterpret_cast<int*>(lg_s + Hq * (T + 1));  // [T][3]

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int v = tid & (L - 1), grp = tid / L;
    constexpr int RS = 256 / L;  // rows per pass
    const bool act = v < NV;
    const int t0_r = grp / H, kh0_r = grp - t0_r * H;  // a lane's first row in a tile
    const int dt_r = RS / H, dkh_r = RS - dt_r * H;     // its step between rows
    const int dt_e = 256 / P, di_e = 256 - dt_e * P;    // cos/sin loop step (t, i)
    const int64_t total = int64_t(a.n_seqs) * a.n_tiles;
    const int64_t t_beg = total * blockIdx.x / gridDim.x, t_end = total * (blockIdx.x + 1) / gridDim.x;
    int cur_b = -1;

    for (int64_t tile = t_beg; tile < t_end; ++tile) {
        const int b = int(tile / a.n_tiles), j = int(tile % a.n_tiles);
        const int m0 = j * T, nt = min(T, M - m0);
        if (b != cur_b) {  // the sequence's raw queries as float32 (4-byte loads)
            const uint32_t* src = reinterpret_cast<const uint32_t*>(a.q + int64_t(b) * Hq * D);
            const int nch = D / 4;
            for (int e = tid; e < Hq * nch; e += blockDim.x) {
                const int hq = e / nch, c = e - hq * nch;
                const uint32_t w0 = src[2 * e], w1 = src[2 * e + 1];
                q_s[((hq % g) * H + hq / g) * qrow + swz(c)] =
                    make_float4(lo_f32(w0), hi_f32(w0), lo_f32(w1), hi_f32(w1));
            }
            cur_b = b;
        }
        const int64_t p = a.q_pos[b];
        const int32_t* crd = a.coords + int64_t(b) * a.coord_seq_stride + 3 * int64_t(m0);
        for (int e = tid; e < 3 * nt; e += blockDim.x) crd_s[e] = crd[e];
        __syncthreads();
        float* cf = reinterpret_cast<float*>(c_s);
        float* sf = reinterpret_cast<float*>(s_s);
        for (int e = tid, t = tid / P, i = tid - (tid / P) * P; e < nt * P;
             e += 256, t += dt_e, i += di_e) {
            if (i >= P) {
                i -= P;
                ++t;
            }
            const int ax = pair_axis(i, a.layout, a.sec_t, a.sec_h, a.sec_w);
            float sn, cn;
            sincos_coord(crd_s[3 * t + ax] - p, a.turn_freq[i], &sn, &cn);
            const int o = (t * crow + swz(i >> 2)) * 4 + (i & 3);
            cf[o] = cn;
            sf[o] = sn;
        }
        __syncthreads();

        const uint16_t* kbase = a.store_k + int64_t(b) * a.store_seq_stride +
                                int64_t(a.layer) * a.store_layer_stride + 8 * v;
        const int rows = nt * H;
        // row r = t * H + kh; a lane's rows advance by RS = dt_r * H + dkh_r.
        // Rows r + RS and r + 2 RS are in flight while row r is computed.
        int t = t0_r, kh = kh0_r;        // the row computed
        int tn = t + dt_r, khn = kh + dkh_r;  // the row two ahead, after the step below
        if (khn >= H) {
            khn -= H;
            ++tn;
        }
        uint4 lo_1 = make_uint4(0, 0, 0, 0), hi_1 = lo_1, lo_2 = lo_1, hi_2 = lo_1;
        if (grp < rows && act) {
            const uint16_t* kr = kbase + int64_t(m0 + t) * a.store_token_stride + kh * D;
            lo_1 = ld_stream(kr);
            hi_1 = ld_stream(kr + P);
        }
        if (grp + RS < rows && act) {
            const uint16_t* kr = kbase + int64_t(m0 + tn) * a.store_token_stride + khn * D;
            lo_2 = ld_stream(kr);
            hi_2 = ld_stream(kr + P);
        }
        for (int r = grp; r - grp < rows; r += RS) {
            const uint4 lo = lo_1, hi = hi_1;
            lo_1 = lo_2;
            hi_1 = hi_2;
            tn += dt_r;
            khn += dkh_r;
            if (khn >= H) {
                khn -= H;
                ++tn;
            }
            if (r + 2 * RS < rows && act) {
                const uint16_t* kr = kbase + int64_t(m0 + tn) * a.store_token_stride + khn * D;
                lo_2 = ld_stream(kr);
                hi_2 = ld_stream(kr + P);
            }
            float acc[G];
#pragma unroll
            for (int h = 0; h < G; ++h) acc[h] = 0.0f;
            if (r < rows && act) {
                const float4* cr = c_s + t * crow;
                const float4* sr = s_s + t * crow;
                const float4 ca = cr[swz(2 * v)], cb = cr[swz(2 * v + 1)];
                const float4 sa = sr[swz(2 * v)], sb = sr[swz(2 * v + 1)];
                const uint32_t lw[4] = {lo.x, lo.y, lo.z, lo.w};
                const uint32_t hw[4] = {hi.x, hi.y, hi.z, hi.w};
                const float2 c2[4] = {make_float2(ca.x, ca.y), make_float2(ca.z, ca.w),
                                      make_float2(cb.x, cb.y), make_float2(cb.z, cb.w)};
                const float2 s2[4] = {make_float2(sa.x, sa.y), make_float2(sa.z, sa.w),
                                      make_float2(sb.x, sb.y), make_float2(sb.z, sb.w)};
                float2 kx[4], ky[4];
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const float2 x = make_float2(__uint_as_float(lw[w] << 16),
                                                 __uint_as_float(lw[w] & 0xffff0000u));
                    const float2 y = make_float2(__uint_as_float(hw[w] << 16),
                                                 __uint_as_float(hw[w] & 0xffff0000u));
                    const float2 ys = __fmul2_rn(y, s2[w]);
                    const float2 xs = __fmul2_rn(x, s2[w]);
                    kx[w] = __ffma2_rn(x, c2[w], make_float2(-ys.x, -ys.y));
                    ky[w] = __ffma2_rn(y, c2[w], xs);
                }
#pragma unroll
                for (int h = 0; h < G; ++h) {
                    if (G != 8 || h < g) {
                        const float4* qr = q_s + (h * H + kh) * qrow;
                        const float4 qa = qr[swz(2 * v)], qb = qr[swz(2 * v + 1)];
                        const float4 qc = qr[swz(P / 4 + 2 * v)], qd = qr[swz(P / 4 + 2 * v + 1)];
                        float2 s2a = __fmul2_rn(make_float2(qa.x, qa.y), kx[0]);
                        s2a = __ffma2_rn(make_float2(qa.z, qa.w), kx[1], s2a);
                        s2a = __ffma2_rn(make_float2(qb.x, qb.y), kx[2], s2a);
                        s2a = __ffma2_rn(make_float2(qb.z, qb.w), kx[3], s2a);
                        s2a = __ffma2_rn(make_float2(qc.x, qc.y), ky[0], s2a);
                        s2a = __ffma2_rn(make_float2(qc.z, qc.w), ky[1], s2a);
                        s2a = __ffma2_rn(make_float2(qd.x, qd.y), ky[2], s2a);
                        s2a = __ffma2_rn(make_float2(qd.z, qd.w), ky[3], s2a);
                        acc[h] = (s2a.x + s2a.y) * a.scale;
                    }
                }
            }
#pragma unroll
            for (int o = L / 2; o; o >>= 1) {
#pragma unroll
                for (int h = 0; h < G; ++h) acc[h] += __shfl_xor_sync(0xffffffffu, acc[h], o);
            }
            if (r < rows && v == 0) {
#pragma unroll
                for (int h = 0; h < G; ++h)
                    if (G != 8 || h < g) lg_s[(kh * g + h) * (T + 1) + t] = acc[h];
            }
            t += dt_r;
            kh += dkh_r;
            if (kh >= H) {
                kh -= H;
                ++t;
            }
        }
        __syncthreads();

        // the tile's logits written out coalesced, a warp per query head
        for (int hq = warp; hq < Hq; hq += blockDim.x >> 5) {
            const float* row = lg_s + hq * (T + 1);
            float* dst = a.logits + (int64_t(b) * Hq + hq) * M + m0;
            for (int t = lane; t < nt; t += 32) dst[t] = row[t];
        }
        // the next tile rewrites the coordinates first, then (after a barrier)
        // the cos/sin rows and logits this tile's warps may still be reading
    }
}

// Tensor-core logits (head_dim 64 and 128). Persistent over work items
// (sequence, group of at most 8 KV heads, 16 NW tokens); warp w of a CTA
// takes tokens 16 w .. 16 w + 15 of the item through the group's KV heads:
//   S (16 rows = the warp's tokens; 8 columns = the GQA group's query heads,
//      columns >= g zero) = K_rot Q^T, D / 8 k-steps of mma.sync m16n8k8 (tf32),
//   K_rot the raw keys turned by the offsets of their coordinates from p.
// The dot product does not depend on the order of the dimensions, so the
// k-slots are permuted: at k-step s, lane group t (= lane & 3) holds pair
// 32 (s / 8) + 8 t + s % 8 of its two tokens (rows g and g + 8), the
// first-half dimension in k-slot t and its rotate-half partner in k-slot
// t + 4. A lane then loads each half of its two rows as 16-byte runs (the
// four lanes of a token cover 64 contiguous bytes) and rotates the two
// tokens' pairs together in packed float2 arithmetic. The cos/sin of a
// lane's (token, pair) are computed once per item into the warp's
// shared-memory table and read back for every KV head. The raw bf16 queries
// are exact tf32 operands (B, kept in shared memory in fragment order per
// (sequence, head group)); each rotated key is split into a tf32 head
// (truncation, one bit operation) and its float32 remainder (< 2^-10 of the
// value, itself truncated by the MMA), and both products are summed in
// float32: ~20 significant bits per product over float32's range. Runs of
// 16-byte loads are double-buffered: the run two ahead is requested as soon
// as a buffer's words are used. Each KV head's logits go straight from the
// accumulators to global memory.
template <int D, int NW>
__global__ void __launch_bounds__(NW * 32, 2) ads_logits_mma_kernel(const __grid_constant__ SelectArgs a) {
    pdl_allow();
    constexpr int P = D / 2, KS = D / 8, NR = KS / 8;  // k-steps; 16-byte runs per half row
    constexpr int T = 16 * NW;                         // tokens per work item
    static_assert(NR == 1 || NR == 2, "head_dim 64 or 128");
    extern __shared__ __align__(16) float sm[];
    const int Hq = a.n_q_heads, H = a.n_kv_heads, g = Hq / H, M = a.n_tokens;
    const int KPI = a.kh_per_item, n_khg = (H + KPI - 1) / KPI;
    const int n_it = (M + T - 1) / T;  // work items per (sequence, head group)
    uint4* qf_s = reinterpret_cast<uint4*>(sm);  // [KPI][KS / 2][32] B fragments
    float4* tr_s = reinterpret_cast<float4*>(qf_s + KPI * (KS / 2) * 32);  // [NW][KS][32]
    uint64_t* tf_s = reinterpret_cast<uint64_t*>(tr_s + NW * KS * 32);      // [P] turn rates
    float2* r8_s = reinterpret_cast<float2*>(tf_s + P);  // [P] turn of 8 w-steps; (1, 0) off the w band
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int gid = lane >> 2, tq = lane & 3;
    for (int i = tid; i < P; i += NW * 32) {
        tf_s[i] = a.turn_freq[i];
        float2 r = make_float2(1.0f, 0.0f);
        if (pair_axis(i, a.layout, a.sec_t, a.sec_h, a.sec_w) == 2) sincos_coord(8, a.turn_freq[i], &r.y, &r.x);
        r8_s[i] = r;
    }
    // axis of this lane's pair at each k-step, two bits each
    uint32_t axes = 0u;
#pragma unroll
    for (int s = 0; s < KS; ++s)
        axes |= uint32_t(pair_axis(32 * (s / 8) + 8 * tq + s % 8, a.layout, a.sec_t, a.sec_h,
                                   a.sec_w)) << (2 * s);
    // the tables above come from the arguments alone: they are set up while
    // the grid this one depends on finishes; every global input is read after
    pdl_wait();
    __syncthreads();
    // Schedule: q = total / grid whole items per CTA, a contiguous run. The
    // R = total - q * grid items left over would make R CTAs run q + 1 items;
    // when 2 R <= grid they are split instead into halves by KV heads, one
    // half per CTA, so that no CTA runs more than q + 1/2 items.
    const int64_t total = int64_t(a.n_seqs) * n_khg * n_it;
    const int64_t G = gridDim.x, q = total / G, R = total - q * G;
    const bool halves = R > 0 && 2 * R <= G && KPI > 1;
    const int64_t c = blockIdx.x;
    const int64_t i_beg = halves ? c * q : total * c / G;
    const int64_t i_end = halves ? i_beg + q : total * (c + 1) / G;
    const int n_work = int(i_end - i_beg) + (halves && c < 2 * R ? 1 : 0);
    int cur_b = -1, cur_kh = -1;
    float4* tr_w = tr_s + warp * KS * 32 + lane;
    const int64_t layer_off = int64_t(a.layer) * a.store_layer_stride + 8 * tq;

    for (int w = 0; w < n_work; ++w) {
        const bool half = i_beg + w >= i_end;
        const int64_t item = half ? q * G + c / 2 : i_beg + w;
        const int64_t bg = item / n_it;  // (sequence, KV-head group)
        const int b = int(bg / n_khg), it = int(item - bg * n_it);
        int kh_a = int(bg - int64_t(b) * n_khg) * KPI, nkh = min(KPI, H - kh_a);
        if (half) {  // the first or second half of the group's KV heads
            const int h1 = (nkh + 1) / 2;
            kh_a += (c & 1) ? h1 : 0;
            nkh = (c & 1) ? nkh - h1 : h1;
        }
        const int j = it * NW + warp;  // the warp's 16-token tile
        const int m0 = 16 * j, ntw = min(16, M - m0);
        // this lane's two tokens (rows g and g + 8 of the warp's MMA tile); a
        // token past the end reads the tile's last token (its logits are
        // never written out)
        const int ta = gid, tb = gid + 8;
        const int ma = m0 + min(ta, ntw - 1), mb = m0 + min(tb, ntw - 1);
        const uint16_t* kb = a.store_k + int64_t(b) * a.store_seq_stride + layer_off;
        const uint16_t* ra = kb + int64_t(ma) * a.store_token_stride;
        const uint16_t* rb = kb + int64_t(mb) * a.store_token_stride;
        const int n_runs = nkh * NR;
        // run r = (KV head kh_a + r / NR, 16-byte run r % NR): first-half x and
        // second-half y words of tokens a and b
        uint4 buf0[4], buf1[4];
        // run u of the KV head whose rows start at pa (token a) and pb (token
        // b): compile-time offsets from two pointers advanced by D per head
        const uint16_t* pa = ra + kh_a * D;
        const uint16_t* pb = rb + kh_a * D;
        auto fetch = [&](uint4 (&k)[4], const uint16_t* xa, const uint16_t* xb, int u) {
            k[0] = ld_stream(xa + 32 * u);
            k[1] = ld_stream(xa + 32 * u + P);
            k[2] = ld_stream(xb + 32 * u);
            k[3] = ld_stream(xb + 32 * u + P);
        };
        if (ntw > 0 && n_runs > 0) {
            fetch(buf0, pa, pb, 0);
            if (NR == 2) fetch(buf1, pa, pb, 1);
            else if (n_runs > 1) fetch(buf1, pa + D, pb + D, 0);
        }
        if (b != cur_b || kh_a != cur_kh) {
            // the group's raw queries as B fragments (a bf16 value is an exact
            // tf32 operand): entry (kh, s / 2, lane) holds k-steps s and s + 1
            __syncthreads();  // every warp is done with the previous group's
            const uint16_t* qs = a.q + int64_t(b) * Hq * D;
            for (int e = tid; e < nkh * (KS / 2) * 32; e += NW * 32) {
                const int kk = e / ((KS / 2) * 32), s2 = (e / 32) % (KS / 2), ln = e & 31;
                const int h = ln >> 2, t4 = ln & 3;
                uint4 f = make_uint4(0u, 0u, 0u, 0u);
                if (h < g) {
                    const uint16_t* qr = qs + ((kh_a + kk) * g + h) * D;
                    const int i0 = 32 * ((2 * s2) / 8) + 8 * t4 + (2 * s2) % 8;  // pair of k-step 2 s2
                    f.x = uint32_t(qr[i0]) << 16;
                    f.y = uint32_t(qr[i0 + P]) << 16;
                    f.z = uint32_t(qr[i0 + 1]) << 16;
                    f.w = uint32_t(qr[i0 + 1 + P]) << 16;
                }
                qf_s[e] = f;
            }
            cur_b = b;
            cur_kh = kh_a;
            __syncthreads();
        }
        if (ntw <= 0 || nkh <= 0) continue;  // past the sequence's last token, or no KV head

        // cos/sin of the lane's (token, pair) at each k-step, at the offsets
        // of the tokens' coordinates from the trigger position
        {
            const int32_t* crd = a.coords + int64_t(b) * a.coord_seq_stride;
            const int64_t p = a.q_pos[b];
            const int ca[3] = {crd[3 * ma], crd[3 * ma + 1], crd[3 * ma + 2]};
            const int cb[3] = {crd[3 * mb], crd[3 * mb + 1], crd[3 * mb + 2]};
            const int64_t oa[3] = {ca[0] - p, ca[1] - p, ca[2] - p};
            // Every lane's two tokens on one image row, 8 columns apart (a
            // 16-token tile within a row): token b's angles are token a's
            // turned by 8 w-steps on the w pairs and equal on the others.
            const bool row8 = __all_sync(0xffffffffu, cb[0] == ca[0] && cb[1] == ca[1] &&
                                                          int64_t(cb[2]) == int64_t(ca[2]) + 8);
            if (row8) {
#pragma unroll
                for (int s = 0; s < KS; ++s) {
                    const uint32_t ax = (axes >> (2 * s)) & 3u;
                    const int i = 32 * (s / 8) + 8 * tq + s % 8;
                    float sn, cs;
                    sincos_coord(ax == 0 ? oa[0] : (ax == 1 ? oa[1] : oa[2]), tf_s[i], &sn, &cs);
                    const float2 r = r8_s[i];
                    tr_w[s * 32] = make_float4(cs, fmaf(cs, r.x, -sn * r.y), sn, fmaf(sn, r.x, cs * r.y));
                }
            } else {
                const int64_t ob[3] = {cb[0] - p, cb[1] - p, cb[2] - p};
#pragma unroll
                for (int s = 0; s < KS; ++s) {
                    const uint32_t ax = (axes >> (2 * s)) & 3u;
                    const uint64_t rate = tf_s[32 * (s / 8) + 8 * tq + s % 8];
                    float4 t;
                    sincos_coord(ax == 0 ? oa[0] : (ax == 1 ? oa[1] : oa[2]), rate, &t.z, &t.x);
                    sincos_coord(ax == 0 ? ob[0] : (ax == 1 ? ob[1] : ob[2]), rate, &t.w, &t.y);
                    tr_w[s * 32] = t;
                }
            }
        }
        __syncwarp();

        float acc[4];
        auto clear = [&]() { acc[0] = acc[1] = acc[2] = acc[3] = 0.0f; };
        clear();
        // the eight k-steps of run u of KV head kk (words in k)
        auto run = [&](const uint4 (&k)[4], int kk, int u) {
            const uint4* qf = qf_s + (kk * (KS / 2) + 4 * u) * 32 + lane;
#pragma unroll
            for (int s8 = 0; s8 < 8; ++s8) {
                const int s = 8 * u + s8, w = s8 / 2;
                const bool up = s8 & 1;  // upper bf16 of the word
                const uint32_t wxa = word_of(k[0], w), wya = word_of(k[1], w);
                const uint32_t wxb = word_of(k[2], w), wyb = word_of(k[3], w);
                const float2 X = up ? make_float2(hi_f32(wxa), hi_f32(wxb))
                                    : make_float2(lo_f32(wxa), lo_f32(wxb));
                const float2 Y = up ? make_float2(hi_f32(wya), hi_f32(wyb))
                                    : make_float2(lo_f32(wya), lo_f32(wyb));
                const float4 t = tr_w[s * 32];
                const float2 C = make_float2(t.x, t.y), S = make_float2(t.z, t.w);
                const float2 ys = __fmul2_rn(Y, S), xs = __fmul2_rn(X, S);
                const float2 Xr = __ffma2_rn(X, C, make_float2(-ys.x, -ys.y));
                const float2 Yr = __ffma2_rn(Y, C, xs);
                // tf32 heads by truncation, float32 remainders
                const uint32_t hxa = __float_as_uint(Xr.x) & 0xffffe000u;
                const uint32_t hxb = __float_as_uint(Xr.y) & 0xffffe000u;
                const uint32_t hya = __float_as_uint(Yr.x) & 0xffffe000u;
                const uint32_t hyb = __float_as_uint(Yr.y) & 0xffffe000u;
                // remainders v - head, two per packed FMA with (-1, -1)
                const float2 lx = __ffma2_rn(make_float2(__uint_as_float(hxa), __uint_as_float(hxb)),
                                             make_float2(-1.0f, -1.0f), Xr);
                const float2 ly = __ffma2_rn(make_float2(__uint_as_float(hya), __uint_as_float(hyb)),
                                             make_float2(-1.0f, -1.0f), Yr);
                const float lxa = lx.x, lxb = lx.y, lya = ly.x, lyb = ly.y;
                const uint4 q2 = qf[(s8 / 2) * 32];
                const uint32_t b0 = up ? q2.z : q2.x, b1 = up ? q2.w : q2.y;
                mma_1688_tf32(acc, hxa, hxb, hya, hyb, b0, b1);
                mma_1688_tf32(acc, __float_as_uint(lxa), __float_as_uint(lxb),
                              __float_as_uint(lya), __float_as_uint(lyb), b0, b1);
            }
        };
        // KV head kk done: its logits out
        const bool va = ta < ntw, vb = tb < ntw;
        // columns 2t, 2t + 1 of each KV head's logits; lg advances by g rows per head
        const int h0 = 2 * tq;
        float* lg = a.logits + (int64_t(b) * Hq + kh_a * g + h0) * M + m0;
        const int64_t lg_step = int64_t(g) * M;
        auto finish = [&]() {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (h0 + c < g) {
                    if (va) lg[int64_t(c) * M + ta] = acc[c] * a.scale;
                    if (vb) lg[int64_t(c) * M + tb] = acc[2 + c] * a.scale;
                }
            }
            lg += lg_step;
            clear();
        };
        // Each buffer's next run is requested as soon as its words are used:
        // head dim 128, buffer u holds run u of the current KV head; head dim
        // 64 (one run per head), buffers take alternate heads.
        if (NR == 2) {
            for (int kk = 0; kk < nkh; ++kk) {
                run(buf0, kk, 0);
                pa += D;
                pb += D;
                if (kk + 1 < nkh) fetch(buf0, pa, pb, 0);
                run(buf1, kk, 1);
                finish();
                if (kk + 1 < nkh) fetch(buf1, pa, pb, 1);
            }
        } else {
            for (int kk = 0; kk < nkh; kk += 2) {
                run(buf0, kk, 0);
                finish();
                if (kk + 2 < nkh) fetch(buf0, pa + 2 * D, pb + 2 * D, 0);
                if (kk + 1 < nkh) {
                    run(buf1, kk + 1, 0);
                    finish();
                    if (kk + 3 < nkh) fetch(buf1, pa + 3 * D, pb + 3 * D, 0);
                }
                pa += 2 * D;
                pb += 2 * D;
            }
        }
    }
}

}  // namespace

size_t select_logits_smem(const SelectArgs& a) {
    const int D = a.head_dim, P = D / 2, T = a.tok_tile;
    return size_t(a.n_q_heads) * (D / 4 + 1) * 16 + 2 * size_t(T) * (P / 4 + 1) * 16 +
           size_t(a.n_q_heads) * (T + 1) * 4 + size_t(T) * 3 * 4;
}

template <int L, int G>
cudaError_t launch_logits_g(const SelectArgs& a, int n_seqs, int sms, cudaStream_t stream) {
    const size_t smem = select_logits_smem(a);
    cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(ads_logits_kernel<L, G>), smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ads_logits_kernel<L, G>, 256, smem);
    if (e != cudaSuccess) return e;
    const int64_t tiles = int64_t(n_seqs) * a.n_tiles;
    const int64_t resident = int64_t(sms) * (per_sm > 0 ? per_sm : 1);
    const unsigned grid = unsigned(tiles < resident ? tiles : resident);
    return launch_pdl(ads_logits_kernel<L, G>, dim3(grid), dim3(256), smem, stream, a);
}

template <int L>
cudaError_t launch_logits(const SelectArgs& a, int n_seqs, int sms, cudaStream_t stream) {
    const int g = a.n_q_heads / a.n_kv_heads;
    if (g == 1) return launch_logits_g<L, 1>(a, n_seqs, sms, stream);
    if (g == 2) return launch_logits_g<L, 2>(a, n_seqs, sms, stream);
    if (g == 4) return launch_logits_g<L, 4>(a, n_seqs, sms, stream);
    return launch_logits_g<L, 8>(a, n_seqs, sms, stream);
}

constexpr int kMmaWarps = 8;  // warps per CTA of the tensor-core logits kernel (16 tokens each)

template <int D>
size_t logits_mma_smem(int kpi) {
    return size_t(kpi) * (D / 16) * 32 * 16 + size_t(kMmaWarps) * (D / 8) * 32 * 16 +
           size_t(D / 2) * 16;
}

template <int D>
cudaError_t launch_logits_mma(const SelectArgs& a, int n_seqs, int sms, cudaStream_t stream) {
    auto kern = ads_logits_mma_kernel<D, kMmaWarps>;
    const int H = a.n_kv_heads;
    SelectArgs b = a;
    b.kh_per_item = H < 8 ? H : 8;  // KV heads per work item (sizes the query fragments)
    const size_t smem_max = logits_mma_smem<D>(b.kh_per_item);
    cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(kern), smem_max);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kMmaWarps * 32, smem_max);
    if (e != cudaSuccess) return e;
    const int64_t resident = int64_t(sms) * (per_sm > 0 ? per_sm : 1);
    // Few tokens (a small batch): fewer KV heads per item until there are two
    // items per resident CTA, so that short chains run side by side.
    const int64_t n_it = (a.n_tokens + 16 * kMmaWarps - 1) / (16 * kMmaWarps);
    auto items = [&](int kpi) { return int64_t(n_seqs) * n_it * ((H + kpi - 1) / kpi); };
    while (b.kh_per_item > 1 && items(b.kh_per_item) < 2 * resident)
        b.kh_per_item = (b.kh_per_item + 1) / 2;
    const int64_t n = items(b.kh_per_item);
    const unsigned grid = unsigned(n < resident ? n : resident);
    return launch_pdl(kern, dim3(grid), dim3(kMmaWarps * 32), logits_mma_smem<D>(b.kh_per_item),
                      stream, b);
}

cudaError_t launch_select(const SelectArgs& a, int n_seqs, int sms, cudaStream_t stream) {
    bool done = false;
    cudaError_t e = launch_select_fused(a, false, n_seqs, sms, stream, &done);
    if (e != cudaSuccess || done) return e;
    const bool mma = (a.head_dim == 128 || a.head_dim == 64) && a.tok_tile == 16;
    if (a.head_dim == 128 && mma) {
        e = launch_logits_mma<128>(a, n_seqs, sms, stream);
    } else if (a.head_dim == 64 && mma) {
        e = launch_logits_mma<64>(a, n_seqs, sms, stream);
    } else {
        const int L = a.head_dim <= 64 ? 4 : (a.head_dim <= 128 ? 8 : 16);
        e = L == 4 ? launch_logits<4>(a, n_seqs, sms, stream)
                   : (L == 8 ? launch_logits<8>(a, n_seqs, sms, stream)
                             : launch_logits<16>(a, n_seqs, sms, stream));
    }
    if (e != cudaSuccess) return e;
    return launch_select_tail(a, n_seqs, !mma, stream);
}

cudaError_t launch_select_cached(const SelectArgs& a, int n_seqs, int sms, cudaStream_t stream) {
    bool done = false;
    cudaError_t e = launch_select_fused(a, true, n_seqs, sms, stream, &done);
    if (e != cudaSuccess || done) return e;
    e = launch_select_cached_logits(a, n_seqs, sms, stream);
    if (e != cudaSuccess) return e;
    return launch_select_tail(a, n_seqs, false, stream);
}

}  // namespace prcr
