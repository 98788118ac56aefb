// First decode step over the active cache (Sec. 3.3, Eq.
// "decode_with_active_cache"): for every sequence, layer and query head,
//   o = softmax(RoPE(q_raw, (p, p, p)) K_act^T / sqrt(D)) V_act
// over the sequence's cache slots [0, len), the revisited rows included.
//
// The step is memory-bound: every cached K/V row is read once. Warps take
// chunks of slots of one KV head of one (sequence, layer) and stream them in
// tiles of 16 slots through tensor cores: at head_dim 64 and 128 (decode_kernel)
// a team of 2 to 12 warps a chunk, or one warp, by decode_chunk's rule; at 256
// (decode_wide_kernel) three. Chunks of one (sequence, layer) are merged by a
// further kernel from (max, sum, accumulator) partials when the sequence is split.
#include <cmath>

#include <cuda_bf16.h>

#include "prcr_device.cuh"
#include "prcr_pdl.cuh"

namespace prcr {
namespace {

constexpr unsigned kFull = 0xffffffffu;
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
                 "r"(src_bytes)
                 : "memory");
}

// Transpose of an 8 x 8 matrix of 16-bit values held as mma fragments
// (lane 4 r + c holds row r, columns 2c and 2c + 1): afterwards the lane holds
// row r, columns 2c and 2c + 1 of the transpose.
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}

// A CTA's warps take consecutive (chunk, KV head) units of one (sequence,
// layer), heads fastest, so that neighbouring warps read neighbouring bytes
// and none idles whatever the head count. Each streams its chunk's tiles
// through a ring of stages in shared memory: K and V by cp.async, the next
// tiles in flight during the current one, the first requested before the
// prologue's barrier (a barrier waits for a thread's plain loads in flight,
// not for its async copies); a lane waits only for its own copies, then a warp
// barrier makes the tile visible. The ring's size bounds the warps per SM
// (DecodeShape): more warps hide more of each warp's latency chain than a
// deeper ring would.
// Per tile (mma.sync m16n8k16, bf16 in, float32 accumulate; g <= 8 query heads
// of the KV head's group):
//   QK:  S^T (16 slots x 8 heads, columns >= g zero) = K (16 slots x 16 dims)
//        x Q^T, D/16 k-steps: the slots fill all 16 MMA rows (with the heads
//        as rows only g of 16 would be used). The dot product does not depend
//        on the order of the dimensions, so lane group t takes 16-byte chunks
//        t, t + 4, ... of its two slots' K rows straight into A fragments;
//        chunk c of slot s is stored at c ^ 4 (s & 1), free of bank conflicts.
//        The query's B fragments stay in registers. Lane (r, t) holds slots r
//        and r + 8 of heads 2t, 2t+1, so it keeps those two heads'
//        online-softmax state (reduced over the eight lanes of one t).
//   PV:  O^T (16 dims x 8 heads) += V^T (16 dims x 16 slots) x P^T (16 slots x
//        8 heads): P^T's B fragments are S^T's 8 x 8 blocks transposed in
//        registers (movmatrix), V's A fragments by ldmatrix.trans from padded
//        rows; O^T's columns are the lane's own heads 2t, 2t+1.
// bf16 operands hold only 8 significant bits, so the float32 query and
// probabilities are split into a bf16 head and a bf16 remainder (two MMAs
// each): products stay exact and the result keeps ~16 bits per operand; K and V
// are bf16 already and enter exactly. A tile's P V is summed from zero and
// added to the running accumulator by the FMA that rescales it.
// TEAM: a CTA of up to kDecodeMaxTeam warps takes one unit, its warps the chunk's
// tiles in turn, and merges their (max, sum, accumulator) in shared memory. A small
// batch mostly needs no chunks and no merge kernel that way (29.2 -> 25.2 us for one
// sequence of 933 slots x 36 layers x 8 heads); a large one at head_dim 128 takes
// teams of four on longer chunks, a quarter of the partials to merge.
// DRAM bounds it: an SM's 12 warps keep ~100 KB in flight (~2.2 us at its share
// of the copy rate). Measured, before | now (before: a CTA looping over the KV
// heads with K in registers for large batches, CTAs of four heads each for
// small ones): 16 sequences x 36 layers x 8 heads of up to 4096 slots 890 | 826
// us, 8 x 28 x 4 212 | 200, 11 x 24 x 5 of up to 6900 554 | 423, 5 x 36 x 8 of up
// to 3500 329 | 287, 14 x 2 x 1 head of up to 7132 37.6 | 19.9; head_dim 64: 12 x
// 28 x 8 275 | 223, 1 x 28 x 4 31.7 | 25.3. Equal static runs of tiles per warp
// instead of chunks: 229 us for the second.
template <int D, bool TEAM>
__global__ void __launch_bounds__(TEAM ? kDecodeMaxTeam * 32 : DecodeShape<D>::kWarps * 32, TEAM ? 1 : DecodeShape<D>::kCtas)
    decode_kernel(const __grid_constant__ DecodeArgs a) {
    const int kRingWarps = TEAM ? int(blockDim.x >> 5) : DecodeShape<D>::kWarps;
    // rounds of eight query pairs per lane: a GQA group is at most 8 heads
    constexpr int kRingQRounds = (D / 2 + 31) / 32;
    constexpr int KS = D / 16;      // k-steps of QK, m-tiles of PV
    constexpr int LV = D / 32;      // 16-byte K chunks per lane per slot
    constexpr int NCH = D / 8;      // 16-byte chunks per row
    constexpr int PITCH = D + 8;    // bf16 per staged V row (pad: conflict-free ldmatrix)
    constexpr int KT = 16 * D;      // bf16 per staged K tile
    constexpr int VT = 16 * PITCH;  // bf16 per staged V tile
    constexpr int NS = DecodeShape<D>::kStages;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(16) float s_cos[kMaxPairs];
    __shared__ __align__(16) float s_sin[kMaxPairs];
    __shared__ uint32_t s_mask[TEAM ? kDecodeMaxTeam : DecodeShape<D>::kWarps][NS];
    __shared__ float s_m[TEAM ? kDecodeMaxTeam : 1][8], s_l[TEAM ? kDecodeMaxTeam : 1][8];
    const int P = D / 2;
    const int g = a.group;
    const int H = a.n_kv_heads;
    const int b = blockIdx.z;
    const int l = blockIdx.y;
    // the ring, stage-major: stage st of warp w holds a K tile then a V tile
    // at ring + (st * kRingWarps + w) * (KT + VT); a warp's rotated queries
    // ([g][D] float32, needed only until it holds its fragments) lie in its
    // share of the last stage, which is first filled after that
    uint16_t* ring = reinterpret_cast<uint16_t*>(smem_raw);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int gid = lane >> 2;
    const int t = lane & 3;
    float* q_s = reinterpret_cast<float*>(ring + size_t((NS - 1) * kRingWarps + warp) * (KT + VT));
    // this warp's (or the team's) chunk and KV head: units of (chunk, head), heads
    // fastest
    const int unit = TEAM ? int(blockIdx.x) : int(blockIdx.x) * kRingWarps + warp;
    const int split = unit / H, kh = unit - split * H;
    const bool wact = split < a.splits;
    const uint16_t* wk = ring + size_t(warp) * (KT + VT);  // this warp's stage 0
    const uint32_t wk_s = uint32_t(__cvta_generic_to_shared(wk));
    const uint32_t wv_s = wk_s + uint32_t(KT * 2);
    const uint32_t kStageBytes = uint32_t(kRingWarps * (KT + VT) * 2);  // one stage of all warps
    uint32_t err = 0;
    const uint16_t* qb = a.q + ((int64_t(b) * a.n_layers + l) * a.n_q_heads + kh * g) * D;
    if (wact)  // the group's query rows into L2 while the preceding grid drains
        for (int o = lane * 64; o < g * D; o += 32 * 64) prefetch_l2(qb + o);
    pdl_wait();
    const int64_t p = a.q_pos[b];
    int64_t len = a.seq_len[b];
    // this lane's query words (eight rotation pairs of a head per round, at
    // most kRingQRounds rounds), requested with the length so that they do not
    // queue behind the ring's first copies
    const bool q16 = (reinterpret_cast<uintptr_t>(a.q) & 15) == 0;
    uint32_t wx[kRingQRounds][4], wy[kRingQRounds][4];
#pragma unroll
    for (int r = 0; r < kRingQRounds; ++r) {
        const int e = 8 * (lane + r * 32);
        if (wact && e < g * P) {
            const int hq = e / P;
            const uint16_t* qx = qb + hq * D + (e - hq * P);
            if (q16) {
                const uint4 x4 = __ldg(reinterpret_cast<const uint4*>(qx));
                const uint4 y4 = __ldg(reinterpret_cast<const uint4*>(qx + P));
                wx[r][0] = x4.x; wx[r][1] = x4.y; wx[r][2] = x4.z; wx[r][3] = x4.w;
                wy[r][0] = y4.x; wy[r][1] = y4.y; wy[r][2] = y4.z; wy[r][3] = y4.w;
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    wx[r][u] = uint32_t(qx[2 * u]) | (uint32_t(qx[2 * u + 1]) << 16);
                    wy[r][u] = uint32_t(qx[P + 2 * u]) | (uint32_t(qx[P + 2 * u + 1]) << 16);
                }
            }
        }
    }
    if (len < 0 || len > a.capacity) {
        err |= PRCR_ST_CAPACITY;
        len = len < 0 ? 0 : a.capacity;
    }
    if (len > int64_t(a.splits) * a.chunk) {  // above the host's max_len: past the split
        err |= PRCR_ST_CAPACITY;
        len = int64_t(a.splits) * a.chunk;
    }
    // A query position beyond the fixed-point angle reduction (|p| >= 2^31)
    // is reported and the sequence attends to nothing: its output is zeros.
    if (p <= -2147483648LL || p >= 2147483648LL) {
        err |= PRCR_ST_POS_RANGE;
        len = 0;
    }
    const int64_t s_begin = int64_t(split) * a.chunk;
    const int64_t s_end = min(len, s_begin + a.chunk);
    // this warp's tiles of the chunk: all of them, or a team's every
    // kRingWarps-th; tile i begins at slot s_begin + i s_step
    const int n_chunk = s_end > s_begin ? int((s_end - s_begin + 15) / 16) : 0;
    const int n_tiles = TEAM ? max(0, (n_chunk - warp + kRingWarps - 1) / kRingWarps) : n_chunk;
    const int64_t s_first = s_begin + (TEAM ? 16 * warp : 0), s_step = TEAM ? 16 * kRingWarps : 16;
    const int64_t lstride = int64_t(l) * a.layer_stride;
    const uint16_t* kbase = a.cache_k + lstride + int64_t(kh) * D;
    const uint16_t* vbase = a.cache_v + lstride + int64_t(kh) * D;

    // block id of this lane's slot (lane & 15) of tile n (paged caches)
    auto block_id = [&](int n) -> int32_t {
        const int64_t s = s_first + s_step * n + (lane & 15);
        if (a.cache_kind != PRCR_CACHE_PAGED || n >= n_tiles || s >= s_end) return 0;
        return a.block_table[int64_t(b) * a.bt_stride + uint32_t(s) / uint32_t(a.block_size)];
    };
    // copies of tile n into stage n % NS (one commit group per call, empty
    // past the last tile or for a warp without a KV head)
    auto issue = [&](int n, int32_t blk) {
        if (wact && n < n_tiles) {
            const int st = n % NS;
            const int64_t s = s_first + s_step * n + (lane & 15);
            int64_t row = -1;
            if (s < s_end) {
                if (a.cache_kind == PRCR_CACHE_CONTIGUOUS) {
                    row = int64_t(b) * a.seq_stride + s * a.slot_stride;
                } else if (blk < 0 || blk >= a.n_blocks) {
                    err |= PRCR_ST_NO_BLOCK;
                } else {
                    row = int64_t(blk) * a.block_stride +
                          int64_t(uint32_t(s) % uint32_t(a.block_size)) * a.slot_stride;
                }
            }
            const uint32_t m = __ballot_sync(kFull, row >= 0) & 0xffffu;
            if (lane == 0) s_mask[warp][st] = m;
            const uint32_t ks_ = wk_s + uint32_t(st) * kStageBytes;
            const uint32_t vs_ = wv_s + uint32_t(st) * kStageBytes;
#pragma unroll
            for (int i = 0; i < (16 * NCH) / 32; ++i) {
                const int c = lane + 32 * i;
                const int slot = c / NCH;
                const int ch = c - slot * NCH;
                const int64_t rr = __shfl_sync(kFull, row, slot);
                const bool ok = rr >= 0;
                cp_async16(ks_ + uint32_t((slot * D + ((ch ^ ((slot & 1) << 2)) * 8)) * 2),
                           ok ? kbase + rr + ch * 8 : kbase, ok ? 16 : 0);
                cp_async16(vs_ + uint32_t((slot * PITCH + ch * 8) * 2),
                           ok ? vbase + rr + ch * 8 : vbase, ok ? 16 : 0);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    // the first NS - 1 tiles are requested now, before the prologue
    {
        int32_t blk[NS - 1];
#pragma unroll
        for (int i = 0; i < NS - 1; ++i) blk[i] = block_id(i);
#pragma unroll
        for (int i = 0; i < NS - 1; ++i) issue(i, blk[i]);
    }
    int32_t blk_next = block_id(NS - 1);

    // the group's query heads rotated at (p, p, p), scaled by 1/sqrt(D): with
    // the same position on every axis, pair i turns by p * inv_freq_i
    // whatever its band, so each pair's cos/sin serves all heads of the CTA
    for (int i = threadIdx.x; i < P; i += blockDim.x)
        sincos_turns(double(p), a.turn_freq[i], &s_sin[i], &s_cos[i]);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRingQRounds; ++r) {
        const int e = 8 * (lane + r * 32);
        if (!wact || e >= g * P) break;
        const int hq = e / P;
        const int i = e - hq * P;  // a multiple of 8: P is 32 or 64
        float rx[8], ry[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float x = __uint_as_float((u & 1) ? (wx[r][u >> 1] & 0xffff0000u) : (wx[r][u >> 1] << 16));
            const float y = __uint_as_float((u & 1) ? (wy[r][u >> 1] & 0xffff0000u) : (wy[r][u >> 1] << 16));
            const float sn = s_sin[i + u], cs = s_cos[i + u];
            rx[u] = fmaf(x, cs, -y * sn) * a.scale;
            ry[u] = fmaf(y, cs, x * sn) * a.scale;
        }
        float4* ox = reinterpret_cast<float4*>(q_s + hq * D + i);
        float4* oy = reinterpret_cast<float4*>(q_s + hq * D + i + P);
        ox[0] = make_float4(rx[0], rx[1], rx[2], rx[3]);
        ox[1] = make_float4(rx[4], rx[5], rx[6], rx[7]);
        oy[0] = make_float4(ry[0], ry[1], ry[2], ry[3]);
        oy[1] = make_float4(ry[4], ry[5], ry[6], ry[7]);
    }
    __syncwarp();

    // the query B fragments (columns = heads of the group; columns >= g are
    // zero); k-step j of lane group t covers dimensions
    // 8 (t + 4 (j / 2)) + 4 (j % 2) + 0..3, as the K chunks it reads
    uint32_t qh[KS][2], ql[KS][2];
    {
        const bool hv = wact && gid < g;
        const float* qr = q_s + (hv ? gid : 0) * D;
#pragma unroll
        for (int j = 0; j < KS; ++j) {
            const float4 x = *reinterpret_cast<const float4*>(qr + 8 * (t + 4 * (j >> 1)) + 4 * (j & 1));
            split_bf16x2(hv ? x.x : 0.0f, hv ? x.y : 0.0f, qh[j][0], ql[j][0]);
            split_bf16x2(hv ? x.z : 0.0f, hv ? x.w : 0.0f, qh[j][1], ql[j][1]);
        }
    }
    __syncwarp();  // the queries' stage may now be filled

    if (wact) {
        float o[KS][4];
#pragma unroll
        for (int mt = 0; mt < KS; ++mt) o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.0f;
        float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.0f, 0.0f};  // heads 2t, 2t + 1
        const int lslot = (lane & 7) + ((lane >> 4) & 1) * 8;
        const int ldim = ((lane >> 3) & 1) * 8;

        for (int n = 0; n < n_tiles; ++n) {
            const int st = n % NS;
            // this lane's copies of tile n are complete; after the warp
            // barrier every lane's are visible
            asm volatile("cp.async.wait_group %0;" ::"n"(NS - 2) : "memory");
            __syncwarp();
            // the tile NS - 1 ahead into the stage tile n - 1 used
            {
                const int32_t bn = blk_next;
                blk_next = block_id(n + NS);
                issue(n + NS - 1, bn);
            }
            const uint32_t mask = s_mask[warp][st];

            const uint16_t* kt = wk + size_t(st) * kRingWarps * (KT + VT);
            // S^T = K Q^T: slots gid and gid + 8 are the A rows; the products of
            // the query's heads and remainders in two chains
            float sh[4] = {0.0f, 0.0f, 0.0f, 0.0f}, sl_[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int u = 0; u < LV; ++u) {
                const int cc = ((t + 4 * u) ^ ((gid & 1) << 2)) * 8;
                const uint4 w0 = *reinterpret_cast<const uint4*>(kt + gid * D + cc);
                const uint4 w1 = *reinterpret_cast<const uint4*>(kt + (gid + 8) * D + cc);
                mma_16816(sh, w0.x, w1.x, w0.y, w1.y, qh[2 * u][0], qh[2 * u][1]);
                mma_16816(sl_, w0.x, w1.x, w0.y, w1.y, ql[2 * u][0], ql[2 * u][1]);
                mma_16816(sh, w0.z, w1.z, w0.w, w1.w, qh[2 * u + 1][0], qh[2 * u + 1][1]);
                mma_16816(sl_, w0.z, w1.z, w0.w, w1.w, ql[2 * u + 1][0], ql[2 * u + 1][1]);
            }

            // online softmax of this lane's heads 2t, 2t + 1 (columns) over the
            // 16 slots: the eight lanes of one t hold them, two slots each
            const bool oka = (mask >> gid) & 1u, okb = (mask >> (8 + gid)) & 1u;
            float pa[2], pb[2], alpha[2];
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const float va = oka ? sh[hh] + sl_[hh] : -INFINITY;
                const float vb = okb ? sh[2 + hh] + sl_[2 + hh] : -INFINITY;
                float mx = fmaxf(va, vb);
                mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 4));
                mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 8));
                mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 16));
                const float m_new = fmaxf(m_run[hh], mx);
                // arguments are <= 0: __expf's error (a few ulp) is far inside
                // that of 16-bit operands
                alpha[hh] = m_new == -INFINITY ? 1.0f : __expf(m_run[hh] - m_new);
                pa[hh] = va == -INFINITY ? 0.0f : __expf(va - m_new);
                pb[hh] = vb == -INFINITY ? 0.0f : __expf(vb - m_new);
                float ps = pa[hh] + pb[hh];
                ps += __shfl_xor_sync(kFull, ps, 4);
                ps += __shfl_xor_sync(kFull, ps, 8);
                ps += __shfl_xor_sync(kFull, ps, 16);
                l_run[hh] = l_run[hh] * alpha[hh] + ps;
                m_run[hh] = m_new;
            }
            // P^T as B fragments: the 8 x 8 blocks (slots 0..7 | 8..15) x heads
            // held as (slot gid; heads 2t, 2t + 1) are transposed in registers
            uint32_t m1h, m1l, m2h, m2l;
            split_bf16x2(pa[0], pa[1], m1h, m1l);
            split_bf16x2(pb[0], pb[1], m2h, m2l);
            const uint32_t pb0h = movmatrix_trans(m1h), pb1h = movmatrix_trans(m2h);
            const uint32_t pb0l = movmatrix_trans(m1l), pb1l = movmatrix_trans(m2l);
            // O^T = alpha O^T + V^T P^T (columns are the lane's own heads)
#pragma unroll
            for (int mt = 0; mt < KS; ++mt) {
                uint32_t r0, r1, r2, r3;
                const uint32_t addr = wv_s + uint32_t(st) * kStageBytes + uint32_t((lslot * PITCH + mt * 16 + ldim) * 2);
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                             : "r"(addr));
                float y[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                mma_16816(y, r0, r1, r2, r3, pb0l, pb1l);
                mma_16816(y, r0, r1, r2, r3, pb0h, pb1h);
                o[mt][0] = fmaf(o[mt][0], alpha[0], y[0]);
                o[mt][1] = fmaf(o[mt][1], alpha[1], y[1]);
                o[mt][2] = fmaf(o[mt][2], alpha[0], y[2]);
                o[mt][3] = fmaf(o[mt][3], alpha[1], y[3]);
            }
            __syncwarp();  // stage st is refilled at the next iteration
        }
        // only now: a following kernel's CTAs, waiting in the room that a grid of one
        // wave leaves, cost its tiles more than an earlier start saved (one sequence
        // of 933 slots x 36 layers x 8 heads 26.9 -> 25.2 us in a row, the pipeline
        // with it and a selection next 56.0 -> 48.8)
        pdl_allow();

        if constexpr (TEAM) {
            // every warp of the CTA is done with its copies: the ring becomes the
            // warps' accumulators
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            float* o_s = reinterpret_cast<float*>(smem_raw) + warp * 8 * (D + 4);
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const int h = 2 * t + hh;
#pragma unroll
                for (int mt = 0; mt < KS; ++mt) {
                    o_s[h * (D + 4) + mt * 16 + gid] = o[mt][hh];
                    o_s[h * (D + 4) + mt * 16 + gid + 8] = o[mt][2 + hh];
                }
                if (gid == 0) {
                    s_m[warp][h] = m_run[hh];
                    s_l[warp][h] = l_run[hh];
                }
            }
            __syncthreads();
            for (int e = threadIdx.x; e < g * (D / 2); e += blockDim.x) {
                const int h = e / (D / 2), d = 2 * (e - h * (D / 2));
                float M = s_m[0][h];
                for (int w = 1; w < kRingWarps; ++w) M = fmaxf(M, s_m[w][h]);
                float2 acc = make_float2(0.0f, 0.0f);
                float den = 0.0f;
                const float* col = reinterpret_cast<const float*>(smem_raw) + h * (D + 4) + d;
                for (int w = 0; w < kRingWarps; ++w) {
                    const float f = s_m[w][h] == -INFINITY ? 0.0f : expf(s_m[w][h] - M);
                    const float2 x = *reinterpret_cast<const float2*>(col + w * 8 * (D + 4));
                    acc.x = fmaf(f, x.x, acc.x);
                    acc.y = fmaf(f, x.y, acc.y);
                    den = fmaf(f, s_l[w][h], den);
                }
                const int64_t o_idx = (int64_t(b) * a.n_layers + l) * a.n_q_heads + kh * g + h;
                if (a.splits == 1) {
                    const float inv = den > 0.0f ? 1.0f / den : 0.0f;
                    *reinterpret_cast<float2*>(a.out + o_idx * D + d) = make_float2(acc.x * inv, acc.y * inv);
                } else {
                    float* part = a.partial + (o_idx * a.splits + split) * (D + 2);
                    *reinterpret_cast<float2*>(part + d) = acc;
                    if (d == 0) *reinterpret_cast<float2*>(part + D) = make_float2(M, den);
                }
            }
        } else {
            // heads 2t, 2t+1 of this lane's O^T columns
            const float l0 = l_run[0], l1 = l_run[1], m0 = m_run[0], m1 = m_run[1];
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const int h = 2 * t + hh;
                if (h >= g) continue;
                const int64_t o_idx = (int64_t(b) * a.n_layers + l) * a.n_q_heads + kh * g + h;
                const float lh = hh ? l1 : l0;
                if (a.splits == 1) {
                    const float inv = lh > 0.0f ? 1.0f / lh : 0.0f;
                    float* out = a.out + o_idx * D;
#pragma unroll
                    for (int mt = 0; mt < KS; ++mt) {
                        out[mt * 16 + gid] = o[mt][hh] * inv;
                        out[mt * 16 + gid + 8] = o[mt][2 + hh] * inv;
                    }
                } else {
                    float* part = a.partial + (o_idx * a.splits + split) * (D + 2);
#pragma unroll
                    for (int mt = 0; mt < KS; ++mt) {
                        part[mt * 16 + gid] = o[mt][hh];
                        part[mt * 16 + gid + 8] = o[mt][2 + hh];
                    }
                    if (gid == 0) {
                        part[D] = hh ? m1 : m0;
                        part[D + 1] = lh;
                    }
                }
            }
        }
    }
    // every copy this thread issued has landed before the CTA may end
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (err) atomicOr(a.status, err);
}

// head_dim 256. A CTA of kWideWarps warps takes one (sequence, layer, KV head,
// chunk); its warps take the chunk's tiles of 16 slots in turn, each through
// its own two-stage shared-memory ring (K and V by cp.async, the next tile in
// flight during the current one), and their (max, sum, accumulator) are
// merged in shared memory at the end.
//   QK:  S^T (16 slots x 8 heads) = K Q^T, 16 k-steps; K's A fragments by
//        ldmatrix from rows padded by 16 bytes (conflict-free).
//   PV:  O^T (256 dims x 8 heads) += V^T P^T, 16 m-tiles, as in the kernels above.
// The float32 query and probabilities enter as three bf16 pieces each (24
// significant bits, three MMAs), the queries' fragments kept in registers
// (96). A tensor core truncates what it adds, so the leading pieces' sums are
// short and start from zero: two k-steps of a logit, one tile of P V, added by
// float32 adds, and by the FMA that rescales the running accumulator; the other
// pieces, 2^-8 as large, are summed apart. Error against float64 over 1..16
// sequences of 64..8192 slots: 1.4e-7 to 2.1e-7 (CUDA-core float32 FMAs 1.8e-7 to
// 5.1e-7; one chain for a tile's P V and two for a logit's sixteen k-steps 2.0e-7
// to 2.7e-7, and slower, each MMA waiting for the last: 813 us for the largest
// below, now 795).
// What bounds it: DRAM. A tile is 16 KB and ~450 warp instructions; an SM's
// share of the copy bandwidth brings a tile in ~745 cycles, in which it can
// issue ~2980. Two CTAs per SM (113 KB of shared memory each) keep six tiles,
// ~100 KB, in flight per SM and hide each other's prologue. Measured against
// the CUDA-core kernel it replaced (one warp per KV head, shuffle-reduced dot
// products, 1.4 TB/s): 16 sequences of up to 4096 slots x 26 layers x 4 KV
// heads (4.9 GB) 3400 -> 795 us, 6.2 TB/s; one of 933 slots 109 -> 29 us.
constexpr int kWideWarps = kDecodeWideWarps;
constexpr int kWideD = 256;
constexpr int kWidePitch = kWideD + 8;           // bf16 per staged row
constexpr int kWideTile = 16 * kWidePitch;       // bf16 per staged K or V tile
constexpr int kWideQPitch = kWideD + 8;          // float32 per rotated query row (conflict-free fragment reads)
constexpr int kWideOPitch = kWideD + 4;          // float32 per merged accumulator row
constexpr size_t kWideSmem = size_t(2) * kWideWarps * 2 * kWideTile * sizeof(uint16_t);
static_assert(8 * kWideQPitch * sizeof(float) <= kWideSmem / 2, "the rotated queries fit in the second stage");
static_assert(kWideWarps * 8 * kWideOPitch * sizeof(float) <= kWideSmem, "the warps' accumulators fit in the ring");

// Two floats as three bf16 pairs whose sum keeps 24 significant bits.
__device__ __forceinline__ void split3_bf16x2(float x0, float x1, uint32_t& h, uint32_t& m, uint32_t& l) {
    h = pack_bf16x2(x0, x1);
    const float r0 = x0 - lo_f32(h), r1 = x1 - hi_f32(h);
    split_bf16x2(r0, r1, m, l);
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

// What the phases of decode_wide_kernel share, in static shared memory.
struct WideShared {
    float cos[kWideD / 2], sin[kWideD / 2];            // of the query's turn
    float m[kWideWarps][8], l[kWideWarps][8];          // every warp's maximum and sum per head
};

// A warp's share of a chunk again, by float32 FMAs, into its accumulators in
// shared memory: for the rare chunk with an infinite or NaN key, value or query. An
// infinity times a zero or negative piece of a split operand is a NaN, where the
// product with the whole operand is an infinity (and a logit of -inf a weight of 0).
// A call, and over the accumulators stored as usual: inlined 801 us for the largest
// shape below, stored in its place 805, this 797, without it 795.
__device__ __noinline__ void wide_exact(const DecodeArgs& a, WideShared& sh, uint32_t s_begin, uint32_t s_end) {
    constexpr int D = kWideD, P = D / 2, V = P / 32;  // a lane has V pairs
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = a.group;
    const int b = blockIdx.z, l = blockIdx.y, kh = int(blockIdx.x) % a.n_kv_heads;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* o_s = reinterpret_cast<float*>(smem_raw) + warp * 8 * kWideOPitch;
    const float *cs = sh.cos, *sn = sh.sin;
    float *m_s = sh.m[warp], *l_s = sh.l[warp];
    const uint16_t* qb = a.q + ((int64_t(b) * a.n_layers + l) * a.n_q_heads + kh * g) * D + lane * V;
    const int64_t head_off = int64_t(l) * a.layer_stride + int64_t(kh) * D + lane * V;
    auto value = [](uint16_t w) { return __uint_as_float(uint32_t(w) << 16); };
    __syncwarp();  // the warp's stores that are overwritten here
    for (int h = 0; h < g; ++h) {
        float qx[V], qy[V], ox[V], oy[V], m = -INFINITY, sum = 0.0f;
        for (int i = 0; i < V; ++i) {
            const float x = value(qb[h * D + i]), y = value(qb[h * D + i + P]), c = cs[lane * V + i], s = sn[lane * V + i];
            qx[i] = fmaf(x, c, -y * s) * a.scale;
            qy[i] = fmaf(y, c, x * s) * a.scale;
            ox[i] = oy[i] = 0.0f;
        }
        for (uint32_t t = s_begin + 16 * warp; t < s_end; t += 16 * kWideWarps) {
            for (uint32_t s = t; s < min(t + 16, s_end); ++s) {
                int64_t row = int64_t(b) * a.seq_stride + int64_t(s) * a.slot_stride;
                if (a.cache_kind == PRCR_CACHE_PAGED) {
                    const int32_t blk = a.block_table[int64_t(b) * a.bt_stride + s / uint32_t(a.block_size)];
                    if (blk < 0 || blk >= a.n_blocks) continue;
                    row = int64_t(blk) * a.block_stride + int64_t(s % uint32_t(a.block_size)) * a.slot_stride;
                }
                const uint16_t* k = a.cache_k + head_off + row;
                const uint16_t* v = a.cache_v + head_off + row;
                float logit = 0.0f;
                for (int i = 0; i < V; ++i) logit = fmaf(qy[i], value(k[i + P]), fmaf(qx[i], value(k[i]), logit));
                for (int o = 16; o; o >>= 1) logit += __shfl_xor_sync(kFull, logit, o);
                const float m_new = fmaxf(m, logit), alpha = m_new == -INFINITY ? 1.0f : expf(m - m_new);
                const float p = logit == -INFINITY ? 0.0f : expf(logit - m_new);
                m = m_new;
                sum = sum * alpha + p;
                for (int i = 0; i < V; ++i) {
                    ox[i] = fmaf(p, value(v[i]), ox[i] * alpha);
                    oy[i] = fmaf(p, value(v[i + P]), oy[i] * alpha);
                }
            }
        }
        for (int i = 0; i < V; ++i) {
            o_s[h * kWideOPitch + lane * V + i] = ox[i];
            o_s[h * kWideOPitch + lane * V + i + P] = oy[i];
        }
        if (lane == 0) {
            m_s[h] = m;
            l_s[h] = sum;
        }
    }
}

__global__ void __launch_bounds__(kWideWarps * 32, 2)
    decode_wide_kernel(const __grid_constant__ DecodeArgs a) {
    constexpr int D = kWideD, P = D / 2, KS = D / 16;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ WideShared sh;
    auto &s_cos = sh.cos, &s_sin = sh.sin;
    auto &s_m = sh.m, &s_l = sh.l;
    const int b = blockIdx.z, l = blockIdx.y, H = a.n_kv_heads, g = a.group;
    const int split = int(blockIdx.x) / H, kh = int(blockIdx.x) - split * H;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, t = lane & 3;
    // the ring, stage-major: stage st of warp w holds a K tile then a V tile;
    // the rotated queries lie in the second stage until every warp holds its
    // fragments
    uint16_t* ring = reinterpret_cast<uint16_t*>(smem_raw);
    float* q_s = reinterpret_cast<float*>(smem_raw + kWideSmem / 2);
    const uint32_t wk_s = uint32_t(__cvta_generic_to_shared(ring + size_t(warp) * 2 * kWideTile));
    constexpr uint32_t kStageBytes = uint32_t(kWideSmem / 2), kTileBytes = uint32_t(kWideTile * 2);
    uint32_t err = 0;
    pdl_wait();
    const int64_t p = a.q_pos[b];
    int64_t len = a.seq_len[b];
    if (len < 0 || len > a.capacity) {
        err |= PRCR_ST_CAPACITY;
        len = len < 0 ? 0 : a.capacity;
    }
    if (len > int64_t(a.splits) * a.chunk) {  // above the host's max_len: past the split
        err |= PRCR_ST_CAPACITY;
        len = int64_t(a.splits) * a.chunk;
    }
    // A query position beyond the fixed-point angle reduction (|p| >= 2^31)
    // is reported and the sequence attends to nothing: its output is zeros.
    if (p <= -2147483648LL || p >= 2147483648LL) {
        err |= PRCR_ST_POS_RANGE;
        len = 0;
    }
    // slots as unsigned 32-bit numbers (seq_len is an int32)
    const uint32_t s_begin = uint32_t(min(int64_t(split) * a.chunk, len));
    const uint32_t s_end = uint32_t(min(len, int64_t(s_begin) + a.chunk));
    const int n_tiles = int((s_end - s_begin + 15) / 16);
    const int64_t head_off = int64_t(l) * a.layer_stride + int64_t(kh) * D;
    const uint16_t* kbase = a.cache_k + head_off + lane * 8;
    const uint16_t* vbase = a.cache_v + head_off + lane * 8;

    // block id of this lane's slot (lane & 15) of tile n (paged caches)
    auto block_id = [&](int n) -> int32_t {
        const uint32_t s = s_begin + uint32_t(16 * n + (lane & 15));
        if (a.cache_kind != PRCR_CACHE_PAGED || s >= s_end) return 0;
        return a.block_table[int64_t(b) * a.bt_stride + s / uint32_t(a.block_size)];
    };
    // copies of tile n into stage st (lane i takes 16-byte chunk i of every
    // row); returns the mask of its readable slots
    auto issue = [&](int n, int st, int32_t blk) -> uint32_t {
        const uint32_t s = s_begin + uint32_t(16 * n + (lane & 15));
        int64_t row = -1;
        if (s < s_end) {
            if (a.cache_kind == PRCR_CACHE_CONTIGUOUS) {
                row = int64_t(b) * a.seq_stride + int64_t(s) * a.slot_stride;
            } else if (blk < 0 || blk >= a.n_blocks) {
                err |= PRCR_ST_NO_BLOCK;
            } else {
                row = int64_t(blk) * a.block_stride +
                      int64_t(s % uint32_t(a.block_size)) * a.slot_stride;
            }
        }
        const uint32_t m = __ballot_sync(kFull, row >= 0) & 0xffffu;
        const uint32_t ks_ = wk_s + uint32_t(st) * kStageBytes + uint32_t(lane * 16);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int64_t rr = __shfl_sync(kFull, row, i);
            const bool ok = rr >= 0;
            cp_async16(ks_ + uint32_t(i * kWidePitch * 2), ok ? kbase + rr : kbase, ok ? 16 : 0);
            cp_async16(ks_ + kTileBytes + uint32_t(i * kWidePitch * 2), ok ? vbase + rr : vbase, ok ? 16 : 0);
        }
        return m;
    };

    // this warp's first tile is requested before the prologue
    uint32_t mask_n = 0u;
    if (warp < n_tiles) mask_n = issue(warp, 0, block_id(warp));
    asm volatile("cp.async.commit_group;" ::: "memory");
    int32_t blk_next = warp + kWideWarps < n_tiles ? block_id(warp + kWideWarps) : 0;

    // the group's query heads rotated at (p, p, p), scaled by 1/sqrt(D)
    for (int i = threadIdx.x; i < P; i += blockDim.x)
        sincos_turns(double(p), a.turn_freq[i], &s_sin[i], &s_cos[i]);
    __syncthreads();
    const uint16_t* qb = a.q + ((int64_t(b) * a.n_layers + l) * a.n_q_heads + kh * g) * D;
    for (int e = threadIdx.x; e < g * (P / 2); e += blockDim.x) {  // two pairs per thread (4-byte loads)
        const int h = e / (P / 2), i = 2 * (e - h * (P / 2));
        const uint32_t wx = __ldg(reinterpret_cast<const unsigned int*>(qb + h * D + i));
        const uint32_t wy = __ldg(reinterpret_cast<const unsigned int*>(qb + h * D + i + P));
        const float c0 = s_cos[i], s0 = s_sin[i], c1 = s_cos[i + 1], s1 = s_sin[i + 1];
        const float x0 = lo_f32(wx), x1 = hi_f32(wx), y0 = lo_f32(wy), y1 = hi_f32(wy);
        *reinterpret_cast<float2*>(q_s + h * kWideQPitch + i) =
            make_float2(fmaf(x0, c0, -y0 * s0) * a.scale, fmaf(x1, c1, -y1 * s1) * a.scale);
        *reinterpret_cast<float2*>(q_s + h * kWideQPitch + i + P) =
            make_float2(fmaf(y0, c0, x0 * s0) * a.scale, fmaf(y1, c1, x1 * s1) * a.scale);
    }
    __syncthreads();
    uint32_t qf[KS][3][2];  // B fragments: column gid = head gid of the group (zero past it)
#pragma unroll
    for (int j = 0; j < KS; ++j) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            float2 x = make_float2(0.0f, 0.0f);
            if (gid < g) x = *reinterpret_cast<const float2*>(q_s + gid * kWideQPitch + 16 * j + 8 * u + 2 * t);
            split3_bf16x2(x.x, x.y, qf[j][0][u], qf[j][1][u], qf[j][2][u]);
        }
    }
    __syncthreads();  // the queries' stage may now be filled

    float o[KS][4];
#pragma unroll
    for (int mt = 0; mt < KS; ++mt) o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.0f;
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.0f, 0.0f};  // heads 2t, 2t + 1
    // ldmatrix row addresses: K (rows = slots), V transposed (rows = slots)
    const uint32_t k_ld = uint32_t(((lane & 15) * kWidePitch + (lane >> 4) * 8) * 2);
    const uint32_t v_ld = kTileBytes + uint32_t((((lane & 7) + ((lane >> 4) & 1) * 8) * kWidePitch + ((lane >> 3) & 1) * 8) * 2);

    int st = 0;
    for (int n = warp; n < n_tiles; n += kWideWarps, st ^= 1) {
        const uint32_t mask = mask_n;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();  // every lane's copies of the tile are visible, and the other stage is read out
        if (n + kWideWarps < n_tiles) {
            const int32_t bn = blk_next;
            blk_next = n + 2 * kWideWarps < n_tiles ? block_id(n + 2 * kWideWarps) : 0;
            mask_n = issue(n + kWideWarps, st ^ 1, bn);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");

        const uint32_t base = wk_s + uint32_t(st) * kStageBytes;
        float c[4][4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u][0] = c[u][1] = c[u][2] = c[u][3] = 0.0f;
#pragma unroll
        for (int j = 0; j < KS; ++j) {
            uint32_t r[4];
            ldmatrix_x4(base + k_ld + uint32_t(j * 32), r);
            if (j & 1) {
                mma_16816(y, r[0], r[1], r[2], r[3], qf[j][0][0], qf[j][0][1]);
#pragma unroll
                for (int u = 0; u < 4; ++u) c[(j >> 1) & 1][u] += y[u];
            } else {
                y[0] = y[1] = y[2] = y[3] = 0.0f;
                mma_16816(y, r[0], r[1], r[2], r[3], qf[j][0][0], qf[j][0][1]);
            }
            mma_16816(c[2], r[0], r[1], r[2], r[3], qf[j][1][0], qf[j][1][1]);
            mma_16816(c[3], r[0], r[1], r[2], r[3], qf[j][2][0], qf[j][2][1]);
        }
        // online softmax of heads 2t, 2t + 1 over slots gid and gid + 8 of the
        // eight lanes of one t
        const bool oka = (mask >> gid) & 1u, okb = (mask >> (8 + gid)) & 1u;
        float pa[2], pb[2], alpha[2];
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const float va = oka ? (c[3][hh] + c[2][hh]) + (c[1][hh] + c[0][hh]) : -INFINITY;
            const float vb = okb ? (c[3][2 + hh] + c[2][2 + hh]) + (c[1][2 + hh] + c[0][2 + hh]) : -INFINITY;
            float mx = fmaxf(va, vb);
            mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 4));
            mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 8));
            mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 16));
            const float m_new = fmaxf(m_run[hh], mx);
            alpha[hh] = m_new == -INFINITY ? 1.0f : expf(m_run[hh] - m_new);
            pa[hh] = va == -INFINITY ? 0.0f : expf(va - m_new);
            pb[hh] = vb == -INFINITY ? 0.0f : expf(vb - m_new);
            float ps = pa[hh] + pb[hh];
            ps += __shfl_xor_sync(kFull, ps, 4);
            ps += __shfl_xor_sync(kFull, ps, 8);
            ps += __shfl_xor_sync(kFull, ps, 16);
            l_run[hh] = l_run[hh] * alpha[hh] + ps;
            m_run[hh] = m_new;
        }
        // P^T as B fragments: the 8 x 8 blocks of S^T transposed in registers
        uint32_t pf[3][2];
        {
            uint32_t w[3];
            split3_bf16x2(pa[0], pa[1], w[0], w[1], w[2]);
#pragma unroll
            for (int u = 0; u < 3; ++u) pf[u][0] = movmatrix_trans(w[u]);
            split3_bf16x2(pb[0], pb[1], w[0], w[1], w[2]);
#pragma unroll
            for (int u = 0; u < 3; ++u) pf[u][1] = movmatrix_trans(w[u]);
        }
        // O^T = alpha O^T + V^T P^T (columns are the lane's own heads)
#pragma unroll
        for (int mt = 0; mt < KS; ++mt) {
            uint32_t r[4];
            ldmatrix_x4_trans(base + v_ld + uint32_t(mt * 32), r);
            float x[4] = {0.0f, 0.0f, 0.0f, 0.0f}, xl[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            mma_16816(xl, r[0], r[1], r[2], r[3], pf[2][0], pf[2][1]);
            mma_16816(xl, r[0], r[1], r[2], r[3], pf[1][0], pf[1][1]);
            mma_16816(x, r[0], r[1], r[2], r[3], pf[0][0], pf[0][1]);
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] += xl[u];
            o[mt][0] = fmaf(o[mt][0], alpha[0], x[0]);
            o[mt][1] = fmaf(o[mt][1], alpha[1], x[1]);
            o[mt][2] = fmaf(o[mt][2], alpha[0], x[2]);
            o[mt][3] = fmaf(o[mt][3], alpha[1], x[3]);
        }
    }

    pdl_allow();  // late, as in decode_kernel
    // merge the warps (the ring is free: no copy is in flight past a warp's last tile)
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    float* o_s = reinterpret_cast<float*>(smem_raw) + warp * 8 * kWideOPitch;
    float any = 0.0f;  // not finite where an accumulator is not
#pragma unroll
    for (int mt = 0; mt < KS; ++mt) any += (o[mt][0] + o[mt][1]) + (o[mt][2] + o[mt][3]);
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
        const int h = 2 * t + hh;
#pragma unroll
        for (int mt = 0; mt < KS; ++mt) {
            o_s[h * kWideOPitch + mt * 16 + gid] = o[mt][hh];
            o_s[h * kWideOPitch + mt * 16 + gid + 8] = o[mt][2 + hh];
        }
        if (gid == 0) {
            s_m[warp][h] = m_run[hh];
            s_l[warp][h] = l_run[hh];
        }
    }
    if (__any_sync(kFull, !(fabsf(any) <= 3.0e38f))) wide_exact(a, sh, s_begin, s_end);
    __syncthreads();
    const float* o_all = reinterpret_cast<const float*>(smem_raw);
    for (int e = threadIdx.x; e < g * (D / 2); e += blockDim.x) {
        const int h = e / (D / 2), d = 2 * (e - h * (D / 2));
        float M = s_m[0][h];
#pragma unroll
        for (int w = 1; w < kWideWarps; ++w) M = fmaxf(M, s_m[w][h]);
        float2 acc = make_float2(0.0f, 0.0f);
        float den = 0.0f;
#pragma unroll
        for (int w = 0; w < kWideWarps; ++w) {
            const float f = s_m[w][h] == -INFINITY ? 0.0f : expf(s_m[w][h] - M);
            const float2 x = *reinterpret_cast<const float2*>(o_all + (w * 8 + h) * kWideOPitch + d);
            acc.x = fmaf(f, x.x, acc.x);
            acc.y = fmaf(f, x.y, acc.y);
            den = fmaf(f, s_l[w][h], den);
        }
        const int64_t o_idx = (int64_t(b) * a.n_layers + l) * a.n_q_heads + kh * g + h;
        if (a.splits == 1) {
            const float inv = den > 0.0f ? 1.0f / den : 0.0f;
            *reinterpret_cast<float2*>(a.out + o_idx * D + d) = make_float2(acc.x * inv, acc.y * inv);
        } else {
            float* part = a.partial + (o_idx * a.splits + split) * (D + 2);
            *reinterpret_cast<float2*>(part + d) = acc;
            if (d == 0) {
                part[D] = M;
                part[D + 1] = den;
            }
        }
    }
    if (err) atomicOr(a.status, err);
}

// Merge the chunks of one (sequence, layer, query head). The chunks' maxima
// and sums are reduced by the whole CTA, their weights exp(m_s - M) staged in
// shared memory 256 at a time, and thread d accumulates dimension d over the
// chunks with eight partial rows requested at once.
__global__ void __launch_bounds__(256) decode_merge_kernel(const __grid_constant__ DecodeArgs a) {
    __shared__ float s_red[8];
    __shared__ float s_w[256];
    const int D = a.head_dim, S = a.splits, R = D + 2;
    pdl_allow();
    pdl_wait();  // the decode grid's partials
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    const int64_t o_idx = blockIdx.x;
    const float* part = a.partial + o_idx * S * R;
    float M = -INFINITY;
    for (int sp = threadIdx.x; sp < S; sp += blockDim.x) M = fmaxf(M, part[int64_t(sp) * R + D]);
#pragma unroll
    for (int o = 16; o; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    if (lane == 0) s_red[warp] = M;
    __syncthreads();
    M = s_red[0];
    for (int w = 1; w < nw; ++w) M = fmaxf(M, s_red[w]);
    __syncthreads();
    float den = 0.0f;
    for (int sp = threadIdx.x; sp < S; sp += blockDim.x) {
        const float ms = part[int64_t(sp) * R + D];
        if (ms != -INFINITY) den = fmaf(expf(ms - M), part[int64_t(sp) * R + D + 1], den);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
    if (lane == 0) s_red[warp] = den;
    __syncthreads();
    den = 0.0f;
    for (int w = 0; w < nw; ++w) den += s_red[w];
    float num[2] = {0.0f, 0.0f};  // dimensions threadIdx.x and threadIdx.x + blockDim.x (D <= 2 x 256)
    for (int s0 = 0; s0 < S; s0 += 256) {
        const int n = min(256, S - s0);
        __syncthreads();
        for (int q = threadIdx.x; q < n; q += blockDim.x) {
            const float ms = part[int64_t(s0 + q) * R + D];
            s_w[q] = ms == -INFINITY ? 0.0f : expf(ms - M);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int d = threadIdx.x + k * blockDim.x;
            if (d >= D) break;
            const float* col = part + int64_t(s0) * R + d;
            float acc = num[k];
            int q = 0;
            for (; q + 8 <= n; q += 8) {
                float x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = col[int64_t(q + u) * R];
#pragma unroll
                for (int u = 0; u < 8; ++u) acc = fmaf(s_w[q + u], x[u], acc);
            }
            for (; q < n; ++q) acc = fmaf(s_w[q], col[int64_t(q) * R], acc);
            num[k] = acc;
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int d = threadIdx.x + k * blockDim.x;
        if (d < D) a.out[o_idx * D + d] = den > 0.0f ? num[k] / den : 0.0f;
    }
}

// Merge for at most 32 chunks: one warp per (sequence, layer, query head).
// Lane s holds chunk s's maximum and sum; the maximum, the weights exp(m_s - M)
// and the denominator stay in registers (shuffles), and lane i accumulates
// dimensions 2i, 2i + 1 (+ 64 k) over the chunks' rows, eight rows at a time. The
// first eight are requested together with the maxima, one round trip for a
// sequence of few chunks: the whole step of one sequence of 933 slots x 36
// layers 29.9 -> 29.2 us.
template <int D>
__global__ void __launch_bounds__(128) decode_merge_warp_kernel(const __grid_constant__ DecodeArgs a,
                                                                int64_t n_out) {
    constexpr int R = D + 2, NV = D / 64;
    pdl_allow();
    pdl_wait();  // the decode grid's partials
    const int S = a.splits;
    const int lane = threadIdx.x & 31;
    const int64_t o_idx = int64_t(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (o_idx >= n_out) return;
    const float* part = a.partial + o_idx * S * R;
    float2 x[8][NV], acc[NV];
    auto load = [&](int s0) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
#pragma unroll
            for (int k = 0; k < NV; ++k)
                x[u][k] = s0 + u < S ? *reinterpret_cast<const float2*>(part + int64_t(s0 + u) * R + 2 * lane + 64 * k)
                                     : make_float2(0.0f, 0.0f);
        }
    };
    load(0);
    const float2 mz = lane < S ? *reinterpret_cast<const float2*>(part + int64_t(lane) * R + D)
                               : make_float2(-INFINITY, 0.0f);
    float M = mz.x;
#pragma unroll
    for (int o = 16; o; o >>= 1) M = fmaxf(M, __shfl_xor_sync(kFull, M, o));
    const float w = mz.x == -INFINITY ? 0.0f : expf(mz.x - M);
    float den = w * mz.y;
#pragma unroll
    for (int o = 16; o; o >>= 1) den += __shfl_xor_sync(kFull, den, o);
    const float inv = den > 0.0f ? 1.0f / den : 0.0f;
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] = make_float2(0.0f, 0.0f);
    for (int s0 = 0; s0 < S; s0 += 8) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float wu = __shfl_sync(kFull, w, (s0 + u) & 31);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                acc[k].x = fmaf(wu, x[u][k].x, acc[k].x);
                acc[k].y = fmaf(wu, x[u][k].y, acc[k].y);
            }
        }
        if (s0 + 8 < S) load(s0 + 8);
    }
#pragma unroll
    for (int k = 0; k < NV; ++k)
        *reinterpret_cast<float2*>(a.out + o_idx * D + 2 * lane + 64 * k) = make_float2(acc[k].x * inv, acc[k].y * inv);
}

template <int D>
cudaError_t launch_d(const DecodeArgs& a, dim3 grid, cudaStream_t stream) {
    using Sh = DecodeShape<D>;
    constexpr size_t per_warp = size_t(Sh::kStages) * 16 * (D + D + 8) * sizeof(uint16_t);
    static_assert(8 * (D + 4) * sizeof(float) <= per_warp, "a team's accumulators fit in its rings");
    const size_t smem = per_warp * (a.team ? a.team : Sh::kWarps);
    static_assert(8 * D * sizeof(float) <= 16 * (2 * D + 8) * sizeof(uint16_t),
                  "a GQA group's rotated queries fit in a warp's share of a ring stage");
    const int64_t units = int64_t(a.splits) * a.n_kv_heads;
    grid.x = unsigned(a.team ? units : (units + Sh::kWarps - 1) / Sh::kWarps);
    auto k = a.team ? decode_kernel<D, true> : decode_kernel<D, false>;
    const cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(k), smem);
    return e != cudaSuccess ? e : launch_pdl(k, grid, dim3((a.team ? a.team : Sh::kWarps) * 32), smem, stream, a);
}

}  // namespace

cudaError_t launch_decode(const DecodeArgs& a, dim3 grid, cudaStream_t stream) {
    cudaError_t e;
    if (a.head_dim == 64) {
        e = launch_d<64>(a, grid, stream);
    } else if (a.head_dim == 128) {
        e = launch_d<128>(a, grid, stream);
    } else {
        // head_dim 256: one KV head per CTA
        dim3 g2 = grid;
        g2.x *= unsigned(a.n_kv_heads);
        e = raise_smem_limit(reinterpret_cast<const void*>(decode_wide_kernel), kWideSmem);
        if (e == cudaSuccess) e = launch_pdl(decode_wide_kernel, g2, dim3(kWideWarps * 32), kWideSmem, stream, a);
    }
    if (e != cudaSuccess || a.splits == 1) return e;
    const int64_t n_out = int64_t(grid.z) * a.n_layers * a.n_q_heads;
    if (a.splits <= 32) {
        auto k = a.head_dim == 64    ? decode_merge_warp_kernel<64>
                 : a.head_dim == 128 ? decode_merge_warp_kernel<128>
                                     : decode_merge_warp_kernel<256>;
        return launch_pdl(k, dim3(unsigned((n_out + 3) / 4)), dim3(128), 0, stream, a, n_out);
    }
    return launch_pdl(decode_merge_kernel, dim3(unsigned(n_out)),
                      dim3(a.head_dim < 256 ? a.head_dim : 256), 0, stream, a);
}

}  // namespace prcr
