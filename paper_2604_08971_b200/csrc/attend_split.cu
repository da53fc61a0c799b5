// SentryAttend (Section 4.4, Eq. 6) for 16-bit tensors in four launches, each of which spreads over the whole GPU:
//
//   score   a warp scores batches of 8 query positions of one (sample, KV group) for all kept heads on the warp MMA, the
//           sampled key rows gathered straight from global memory (they stay in L1: no staging, no barriers); the block
//           also lists the sample's present tokens and sums V over its positions
//   select  the U best positions per head, a warp (T <= 1024) or a block each
//   rows    Eq. 6 on tiles of 16 active rows, a warp per tile and part of the keys, K and V fragments from global memory
//   fill    context and zero rows, and the merge of the key parts
//
// A CTA per (sample, group) does the same in attend_bf16.cu and attend_long.cu: ten phases with a barrier after each, of
// which every one is a chain of latencies, on as many SMs as there are groups.  Taken apart, each phase runs with as many
// warps as it has work: the form for long sequences and for few groups (attend_split_faster in api.cu has the line).
// Measured on 16 x 4096 tokens, d = 32, 4 of 8 heads kept: 310 us before, 91 as four launches (100 with the parts of Eq. 6
// merged by one warp per tile and the token list read twice).
#include <math.h>
#include <stddef.h>

#include "attend_common.cuh"

namespace {

constexpr int kSplitThreads = 256, kSplitWarps = kSplitThreads / 32;
constexpr int kScoreBlock = 128;                 // query positions per score block
constexpr int kRowTiles = kMaxRK * kMaxActive / 16;
constexpr int kMaxParts = 16;                     // parts of the keys in the rows launch

// ------------------------------------------------------------------------------------------ pieces
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// The D/8 words of a row that lane quarter tq holds as an MMA operand, straight from global memory: the K index of the
// MMA is permuted so that they are contiguous (d = 16: 8 bytes, 32: 16 bytes, 64: pieces tq and tq + 4 of 16 bytes); key and
// query fragments use the same order.
template <int D>
__device__ __forceinline__ void ld_row_frag(uint32_t (&w)[D / 8], const __nv_bfloat16* row, int tq) {
    if constexpr (D == 16) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(row) + tq);
        w[0] = v.x; w[1] = v.y;
    } else {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(row) + tq);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
        if constexpr (D == 64) {
            const uint4 u = __ldg(reinterpret_cast<const uint4*>(row) + 4 + tq);
            w[4] = u.x; w[5] = u.y; w[6] = u.z; w[7] = u.w;
        }
    }
}
// c0, c1 = rows 0..7 of the 16 x 8 x D product (rows 8..15 of A are zero and their results dropped)
template <int D>
__device__ __forceinline__ void mma_rows8(float& c0, float& c1, const uint32_t (&q)[D / 8], const uint32_t (&k)[D / 8]) {
    float c2, c3;
    asm("mma.sync.aligned.m16n8k16.row.col.f32." ATT_PTX_TYPE "." ATT_PTX_TYPE ".f32 {%0, %1, %2, %3}, {%4, %6, %5, %6}, "
        "{%7, %8}, {%9, %9, %9, %9};"
        : "=f"(c0), "=f"(c1), "=f"(c2), "=f"(c3) : "r"(q[0]), "r"(q[1]), "r"(0), "r"(k[0]), "r"(k[1]), "f"(0.f));
#pragma unroll
    for (int ks = 1; ks < D / 16; ++ks)
        asm("mma.sync.aligned.m16n8k16.row.col.f32." ATT_PTX_TYPE "." ATT_PTX_TYPE ".f32 {%0, %1, %2, %3}, {%4, %6, %5, %6}, "
            "{%7, %8}, {%0, %1, %2, %3};"
            : "+f"(c0), "+f"(c1), "+f"(c2), "+f"(c3) : "r"(q[2 * ks]), "r"(q[2 * ks + 1]), "r"(0), "r"(k[2 * ks]), "r"(k[2 * ks + 1]));
}

// Present-token list of a sample, ascending, by 256 threads: every warp a run of 32-token pieces, after one count of what
// comes before it.  red: kSplitWarps ints.  Returns T_v; the list is complete behind the caller's next barrier.
__device__ __forceinline__ int list_present(const int32_t* __restrict__ ids, int T, uint32_t mask, uint16_t* valid, int* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int pieces = (T + 31) / 32, per = (pieces + kSplitWarps - 1) / kSplitWarps;
    const int p0 = min(warp * per, pieces), p1 = min(p0 + per, pieces);
    auto present = [&](int t) {
        const int m = t < T ? __ldg(ids + t) : -1;
        return m >= 0 && m < 32 && ((mask >> m) & 1u);
    };
    constexpr int HELD = 8;       // ballots of the run's first pieces stay in registers (all of it up to T = 2048; 16 cost more)
    unsigned bm[HELD];
    int mine = 0;
    {
        bool ok[HELD];
#pragma unroll
        for (int j = 0; j < HELD; ++j) ok[j] = p0 + j < p1 && present((p0 + j) * 32 + lane);   // all loads on the way at once
#pragma unroll
        for (int j = 0; j < HELD; ++j) { bm[j] = __ballot_sync(0xffffffffu, ok[j]); mine += __popc(bm[j]); }
    }
#pragma unroll 4
    for (int pc = p0 + HELD; pc < p1; ++pc) mine += __popc(__ballot_sync(0xffffffffu, present(pc * 32 + lane)));
    if (lane == 0) red[warp] = mine;
    __syncthreads();
    int base = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kSplitWarps; ++w) { const int c = red[w]; total += c; if (w < warp) base += c; }
    auto put = [&](int pc, unsigned m) {
        if ((m >> lane) & 1u) valid[base + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(pc * 32 + lane);
        base += __popc(m);
    };
#pragma unroll
    for (int j = 0; j < HELD; ++j) put(p0 + j, bm[j]);
#pragma unroll 4
    for (int pc = p0 + HELD; pc < p1; ++pc) put(pc, __ballot_sync(0xffffffffu, present(pc * 32 + lane)));
    return total;
}

// The kept heads of group g by one warp: ids to hs, kept-list slots to khs (shared, kMaxRK each), count returned.
__device__ __forceinline__ int warp_group_heads(const int32_t* kept_row, int k_h, int r, int g, int Hq, int* hs, int* khs, bool& bad) {
    const int lane = threadIdx.x & 31;
    int rk = 0;
    bad = false;
    for (int j0 = 0; j0 < k_h; j0 += 32) {
        const int j = j0 + lane;
        const int h = j < k_h ? kept_row[j] : -1;
        if (j < k_h && (h < 0 || h >= Hq)) bad = true;
        const bool in = h >= 0 && h < Hq && h / r == g;
        const unsigned im = __ballot_sync(0xffffffffu, in);
        const int at = rk + __popc(im & ((1u << lane) - 1u));
        if (in && at < kMaxRK) { hs[at] = h; khs[at] = j; }
        rk += __popc(im);
    }
    return min(rk, kMaxRK);
}

// Where the sampled key positions of a query come from.
struct SampleSrc {
    const int32_t* tbl;   // table of the sample's subset (null in score_mode 1)
    int n_s;              // sampled keys per query
    int cnt;              // keys a query is scored on: n_s, or T_v in score_mode 1
    int score_mode;
    __device__ __forceinline__ int at(int p, int a, int Tv) const {
        return score_mode == 1 ? a : __ldg(tbl + (score_mode == 2 ? (size_t)a * Tv + p : (size_t)p * n_s + a));
    }
};

struct SplitArgs {
    const __nv_bfloat16 *Q, *K, *V;
    const int32_t* kept_heads;
    const int32_t* ids;
    const uint32_t* masks;
    const int32_t* table;
    const int64_t* offsets;
    int n_subsets, B, T, Hq, Hk, k_h, c, score_mode, U_max, nsplit, n_blk;
    bool given;                   // `active` is the caller's selection
    const float* gate_scores;     // head selection in the score launch (null: kept_heads is given)
    int gate_S;
    int32_t* kept_out;
    float* mscore;                // [B, k_h, T]
    uint16_t* valid;              // [B, T] present tokens
    int* tv;                      // [B]
    float* vsum;                  // [B, Hk, n_blk, D] column sums of V over the positions of a score block
    float* part;                  // [B, Hk, nsplit, kRowTiles, 32 lanes, D/2 + 4] parts of Eq. 6 (nsplit > 1)
    int32_t* active;              // [B, k_h, U_max]
    __nv_bfloat16* O;
    unsigned int* status;
};

// ------------------------------------------------------------------------------------------ score
// Max and sum of the scores of the lane's row over NT tiles of 8 sampled keys; idx: this lane's first staged token.
// tail: valid columns of the last tile counted from this lane's first.
template <int D, int NT>
__device__ __forceinline__ void score_query(const uint32_t (&qf)[D / 8], const __nv_bfloat16* Kg, const uint16_t* idx, int tq,
                                            int tail, float& mx, float& sm) {
    mx = -INFINITY;
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        uint32_t kf[D / 8];
        ld_row_frag<D>(kf, Kg + (uint32_t)idx[t * 8] * D, tq);
        float c0, c1;
        mma_rows8<D>(c0, c1, qf, kf);
        mx = max3(mx, c0, c1);
        if (t == NT - 1) {
            c0 = tail > 0 ? c0 : 0.f;
            c1 = tail > 1 ? c1 : 0.f;
        }
        s0 += c0;
        s1 += c1;
    }
    sm = s0 + s1;
}

// The rows of several queries sit in the A operand together (8 / kept heads of them): a tile of sampled keys belongs to
// one of them, the lanes of the other rows drop theirs, and the query fragment and the reduction across lanes are paid
// once per set.  NT = key tiles per query (0: every present key, no table).
template <int D, int NT>
__device__ __forceinline__ void score_batches(const __nv_bfloat16* __restrict__ qh, const __nv_bfloat16* __restrict__ Kg,
                                              float* __restrict__ out, bool mine, int lh, const uint16_t* s_valid,
                                              uint16_t* s_idx, int Tv, int p_begin, int p_end, const SampleSrc& src, int warp,
                                              unsigned int* status) {
    constexpr int W = D / 8;
    const int lane = threadIdx.x & 31, gq = lane >> 2, tq = lane & 3;
    const int my_j = gq >> lh, QP = 8 >> lh;
    const float scale = rsqrtf((float)D), inv_cnt = 1.0f / (float)src.cnt;
    for (int p0 = p_begin + warp * 8; p0 < p_end; p0 += kSplitWarps * 8) {
        if constexpr (NT > 0) {
            // 8 queries x 8 NT sampled positions -> tokens; entries past the count repeat the last one
            const int q = lane & 7, a4 = lane >> 3, p = min(p0 + q, Tv - 1);
            const int first = src.score_mode == 2 ? p : p * src.n_s, es = src.score_mode == 2 ? Tv : 1;
            int e[2 * NT];
#pragma unroll
            for (int i = 0; i < 2 * NT; ++i) {
                const int at = i < 2 * NT - 2 ? 4 * i + a4 : min(4 * i + a4, src.cnt - 1);
                e[i] = __ldg(src.tbl + (first + at * es));
            }
            bool bad = false;
#pragma unroll
            for (int i = 0; i < 2 * NT; ++i) {
                if ((unsigned)e[i] >= (unsigned)Tv) { bad = true; e[i] = 0; }
                s_idx[q * NT * 8 + 4 * i + a4] = s_valid[e[i]];
            }
            if (bad) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
            __syncwarp();
        }
#pragma unroll 1
        for (int j0 = 0; j0 < 8 && p0 + j0 < p_end; j0 += QP) {
            uint32_t qf[W];
#pragma unroll
            for (int i = 0; i < W; ++i) qf[i] = 0u;
            const int pq = p0 + j0 + my_j;
            if (mine && pq < p_end) ld_row_frag<D>(qf, qh + (uint32_t)s_valid[pq] * D, tq);
            float M = -INFINITY, Sm = 0.f;
            if constexpr (NT > 0) {
                const int nq = min(QP, p_end - p0 - j0);
                const uint16_t* my_idx = s_idx + j0 * NT * 8 + gq;
                const int tail = src.cnt - (NT - 1) * 8 - 2 * tq;
#pragma unroll 1
                for (int j = 0; j < nq; ++j, my_idx += NT * 8) {
                    float mx, sm;
                    score_query<D, NT>(qf, Kg, my_idx, tq, tail, mx, sm);
                    if (my_j == j) { M = mx; Sm = sm; }
                }
            } else {
                // all present keys: the same key tiles for every query row, so one walk serves the whole set
                for (int t = 0; t * 8 < Tv; ++t) {
                    uint32_t kf[W];
                    ld_row_frag<D>(kf, Kg + (uint32_t)s_valid[min(t * 8 + gq, Tv - 1)] * D, tq);
                    float c0, c1;
                    mma_rows8<D>(c0, c1, qf, kf);
                    M = max3(M, c0, t * 8 + 2 * tq + 1 < Tv ? c1 : c0);
                    if (t * 8 + 2 * tq < Tv) Sm += c0;
                    if (t * 8 + 2 * tq + 1 < Tv) Sm += c1;
                }
            }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
                Sm += __shfl_xor_sync(0xffffffffu, Sm, o);
            }
            if (mine && tq == 0 && pq < p_end) out[pq] = (M - Sm * inv_cnt) * scale;
        }
        __syncwarp();   // the staged positions are free for the next batch
    }
}

// grid B * Hk * n_blk (blocks of a group together).  Dynamic smem: valid[T] u16 | staged tokens of the warps' batches.
// Bound by the L1's gathers of key rows, 16 bytes a lane: with four lanes to a 64-byte row they take 6 cycles a warp.  128
// query positions per block: a batch of 8 for every warp twice, which leaves 4 blocks per SM at 16 x 4096.
template <int D>
__global__ void __launch_bounds__(kSplitThreads, 4)
attend_split_score_kernel(const __grid_constant__ SplitArgs a) {
    extern __shared__ __align__(128) uint8_t s_raw[];
    __shared__ int red[kSplitWarps], s_hs[kMaxRK], s_khs[kMaxRK], s_rk;
    __shared__ int32_t s_kept[64];
    __shared__ float s_vs[kSplitWarps][D];
    uint16_t* s_valid = reinterpret_cast<uint16_t*>(s_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint16_t* s_idx = s_valid + ((a.T + 63) & ~63) + warp * 8 * kMaxActive;
    const int grp = blockIdx.x / a.n_blk, blk = blockIdx.x % a.n_blk;
    const int b = grp / a.Hk, g = grp % a.Hk;
    grid_dependency_wait();
    const uint32_t mask = a.masks[b];
    if (warp == 0) {
        const int32_t* kept_row = a.kept_heads + (size_t)b * a.k_h;
        if (a.gate_scores != nullptr) {
            // SentryGate's head selection for this sample's mask: the k_h best of the Hq <= 64 scores of row `mask` (score
            // descending, equal scores -> lower index, NaN below every number), ascending.  Every block of the sample
            // computes the same list; one leaves it in kept_out.
            const unsigned lt = (1u << lane) - 1u;
            uint32_t row = mask;
            if (row >= (uint32_t)a.gate_S) { if (lane == 0) atomicOr(a.status, SENTRY_STATUS_BIT_BAD_INDEX); row = 0; }
            const float* sr = a.gate_scores + (size_t)row * a.Hq;
            const uint32_t k0 = lane < a.Hq ? sentry_order_key(sr[lane]) : 0u;
            const uint32_t k1 = lane + 32 < a.Hq ? sentry_order_key(sr[lane + 32]) : 0u;
            int r0 = 0, r1 = 0;
            for (int j = 0; j < a.Hq; ++j) {
                const uint32_t kj = __shfl_sync(0xffffffffu, j < 32 ? k0 : k1, j & 31);
                r0 += (kj > k0 || (kj == k0 && j < lane)) ? 1 : 0;
                r1 += (kj > k1 || (kj == k1 && j < lane + 32)) ? 1 : 0;
            }
            const bool keep0 = lane < a.Hq && r0 < a.k_h, keep1 = lane + 32 < a.Hq && r1 < a.k_h;
            const unsigned b0 = __ballot_sync(0xffffffffu, keep0), b1 = __ballot_sync(0xffffffffu, keep1);
            if (keep0) s_kept[__popc(b0 & lt)] = lane;
            if (keep1) s_kept[__popc(b0) + __popc(b1 & lt)] = lane + 32;
            __syncwarp();
            if (g == 0 && blk == 0)
                for (int i = lane; i < a.k_h; i += 32) a.kept_out[(size_t)b * a.k_h + i] = s_kept[i];
            kept_row = s_kept;
        }
        bool bad;
        const int n = warp_group_heads(kept_row, a.k_h, a.Hq / a.Hk, g, a.Hq, s_hs, s_khs, bad);
        if (bad && blk == 0) atomicOr(a.status, SENTRY_STATUS_BIT_BAD_INDEX);
        if (lane == 0) s_rk = n;
    }
    const int Tv = list_present(a.ids, a.T, mask, s_valid, red);
    __syncthreads();
    const int rk = s_rk;
    const int p_begin = blk * kScoreBlock, p_end = min(Tv, p_begin + kScoreBlock);
    if (g == 0) {   // the list for the launches that follow
        for (int p = p_begin + threadIdx.x; p < p_end; p += kSplitThreads) a.valid[(size_t)b * a.T + p] = s_valid[p];
        if (blk == 0 && threadIdx.x == 0) a.tv[b] = Tv;
    }
    if (rk == 0) return;
    if (Tv == 0 && blk == 0 && threadIdx.x == 0) atomicOr(a.status, SENTRY_STATUS_BIT_EMPTY_MASK);
    if (p_begin >= Tv) return;
    {   // column sums of V over this block's positions: 16 bytes of a row per lane
        constexpr int CPR = D / 8, RPW = 32 / CPR;
        const __nv_bfloat16* Vg = a.V + (size_t)grp * a.T * D;
        const int cc = lane % CPR;
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = 0.f;
#pragma unroll 2
        for (int p = p_begin + warp * RPW + lane / CPR; p < p_end; p += kSplitWarps * RPW) {
            const uint4 w = __ldg(reinterpret_cast<const uint4*>(Vg + (size_t)s_valid[p] * D) + cc);
            v[0] += att_lo(w.x); v[1] += att_hi(w.x); v[2] += att_lo(w.y); v[3] += att_hi(w.y);
            v[4] += att_lo(w.z); v[5] += att_hi(w.z); v[6] += att_lo(w.w); v[7] += att_hi(w.w);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e)
#pragma unroll
            for (int o = CPR; o < 32; o <<= 1) v[e] += __shfl_xor_sync(0xffffffffu, v[e], o);
        if (lane < CPR) {
#pragma unroll
            for (int e = 0; e < 8; ++e) s_vs[warp][cc * 8 + e] = v[e];
        }
    }
    __syncthreads();
    if (threadIdx.x < D) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < kSplitWarps; ++w) t += s_vs[w][threadIdx.x];
        a.vsum[((size_t)grp * a.n_blk + blk) * D + threadIdx.x] = t;
    }
    if (a.given) return;

    const int lh = rk == 1 ? 0 : (rk == 2 ? 1 : 2);   // log2 of the padded head count
    const int my_h = (lane >> 2) & ((1 << lh) - 1);
    const bool mine = my_h < rk;
    const int hq = s_hs[min(my_h, rk - 1)], kh = s_khs[min(my_h, rk - 1)];
    const __nv_bfloat16* qh = a.Q + ((size_t)b * a.Hq + hq) * a.T * D;
    const __nv_bfloat16* Kg = a.K + (size_t)grp * a.T * D;
    float* out = a.mscore + ((size_t)b * a.k_h + kh) * a.T;
    SampleSrc src;
    src.score_mode = a.score_mode;
    src.n_s = sentry_num_active(Tv, a.c);
    src.cnt = a.score_mode != 1 ? src.n_s : Tv;
    src.tbl = nullptr;
    if (a.score_mode != 1) {
        if (mask >= (uint32_t)a.n_subsets || a.offsets[mask] < 0) {   // no table: every score ties
            if (threadIdx.x == 0) atomicOr(a.status, SENTRY_STATUS_BIT_BAD_INDEX);
            for (int h = 0; h < rk; ++h)
                for (int p = p_begin + threadIdx.x; p < p_end; p += kSplitThreads)
                    a.mscore[((size_t)b * a.k_h + s_khs[h]) * a.T + p] = 0.f;
            return;
        }
        src.tbl = a.table + a.offsets[mask];
    }
#define SCORE_CASE(N) score_batches<D, N>(qh, Kg, out, mine, lh, s_valid, s_idx, Tv, p_begin, p_end, src, warp, a.status)
    switch (a.score_mode == 1 ? 0 : (src.cnt + 7) >> 3) {
        case 0: SCORE_CASE(0); break;
        case 1: SCORE_CASE(1); break;
        case 2: SCORE_CASE(2); break;
        case 3: SCORE_CASE(3); break;
        case 4: SCORE_CASE(4); break;
        case 5: SCORE_CASE(5); break;
        default: SCORE_CASE(6); break;
    }
#undef SCORE_CASE
}

// ------------------------------------------------------------------------------------------ select
// The MMA sums in its own order, so a score may differ from an fp32 loop's over the table row by rounding.  The selection
// takes the scores as approximate: entries within a margin of the U-th score are scored again in the loop's order and
// ranked on that, so that what is selected does not depend on which kernel computed the scores.  Most heads have no
// contested entry.
//
// The score of one query position in the order of the loop, by a whole warp: every lane takes one sampled key, the sum
// then runs over the lanes in table order.
template <int D>
__device__ __noinline__ uint32_t exact_score_key(const __nv_bfloat16* qrow, const __nv_bfloat16* Kg, const uint16_t* valid,
                                                 int Tv, SampleSrc src, int p) {
    const int lane = threadIdx.x & 31;
    const float scale = rsqrtf((float)D);
    float mx = -INFINITY, sum = 0.f;
    for (int a0 = 0; a0 < src.cnt; a0 += 32) {
        const int at = min(a0 + lane, src.cnt - 1);
        int pj = src.at(p, at, Tv);
        if (pj < 0 || pj >= Tv) pj = 0;
        const uint4* kr = reinterpret_cast<const uint4*>(Kg + (size_t)valid[pj] * D);
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int cc = 0; cc < D / 8; ++cc) {
            const uint4 q = __ldg(reinterpret_cast<const uint4*>(qrow) + cc), v = __ldg(kr + cc);
            fma_bf16_pair(acc[0], acc[1], q.x, v.x);
            fma_bf16_pair(acc[2], acc[3], q.y, v.y);
            fma_bf16_pair(acc[0], acc[1], q.z, v.z);
            fma_bf16_pair(acc[2], acc[3], q.w, v.w);
        }
        const float sc = ((acc[0] + acc[1]) + (acc[2] + acc[3])) * scale;
        const int n = min(32, src.cnt - a0);
        for (int j = 0; j < n; ++j) {
            const float v = __shfl_sync(0xffffffffu, sc, j);
            mx = fmaxf(mx, v);
            sum += v;
        }
    }
    return sentry_order_key(mx - sum * (1.0f / (float)src.cnt));
}

__device__ __forceinline__ float order_key_value(uint32_t key) {   // inverse of sentry_order_key (not for NaN's 0)
    return __uint_as_float((key & 0x80000000u) ? (key ^ 0x80000000u) : ~key);
}
// Margin within which two approximate scores are not taken to be in order, as a fraction of the head's largest |M|.
// The fp32 loop and the MMA each round to about 1e-6 of sum |q_i k_i| / sqrt d, which is 1 to 3 times the largest score for
// data without systematic cancellation; measured differences are a tenth of that.
constexpr float kScoreMargin = 1.0f / 262144.0f;

// Sum, max or min of a value over the NW warps that share a head (NW = 1: over the lanes).  buf: which of two exchange
// buffers in turn -- the barrier of one exchange also frees the buffer of the one before.
template <int NW>
struct HeadReduce {
    uint32_t (*x)[3][8];
    int buf, lane, warp;
    __device__ __forceinline__ void sum3(uint32_t& p, uint32_t& q) {
        p = __reduce_add_sync(0xffffffffu, p);
        q = __reduce_add_sync(0xffffffffu, q);
        if constexpr (NW > 1) {
            if (lane == 0) { x[buf][0][warp] = p; x[buf][1][warp] = q; }
            __syncthreads();
            p = q = 0u;
#pragma unroll
            for (int w = 0; w < NW; ++w) { p += x[buf][0][w]; q += x[buf][1][w]; }
            buf ^= 1;
        }
    }
    __device__ __forceinline__ void max_min(uint32_t& p, uint32_t& q) {
        p = __reduce_max_sync(0xffffffffu, p);
        q = __reduce_min_sync(0xffffffffu, q);
        if constexpr (NW > 1) {
            if (lane == 0) { x[buf][0][warp] = p; x[buf][1][warp] = q; }
            __syncthreads();
#pragma unroll
            for (int w = 0; w < NW; ++w) { p = max(p, x[buf][0][w]); q = min(q, x[buf][1][w]); }
            buf ^= 1;
        }
    }
};

// The U best of a head's T_v scores (larger first, ties -> lower position) as ascending tokens: KPT consecutive keys per
// lane in registers, NW warps per head (1: eight heads per block, 8: a block per head).  The threshold is found two bits
// per step -- three candidates counted at once -- from the first bit in which the keys differ until exactly U keys lie
// above one: 6 to 8 steps.  Bound by latency: a warp-wide reduction takes 56 cycles, a block-wide round 300.
template <int D, int KPT, int NW>
__global__ void __launch_bounds__(kSplitThreads)
attend_split_select_kernel(const __grid_constant__ SplitArgs a) {
    __shared__ uint32_t s_x[2][3][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wi = NW == 1 ? 0 : warp;
    grid_dependency_wait();
    const int hidx = NW == 1 ? (int)blockIdx.x * kSplitWarps + warp : (int)blockIdx.x;
    if (hidx >= a.B * a.k_h) return;
    const int b = hidx / a.k_h;
    const int Tv = a.tv[b], h = a.kept_heads[hidx], U = sentry_num_active(Tv, a.c);
    int32_t* out = a.active + (size_t)hidx * a.U_max;
    const bool dead = Tv == 0 || h < 0 || h >= a.Hq;
    for (int i = (dead ? 0 : U) + wi * 32 + lane; i < a.U_max; i += NW * 32) out[i] = -1;
    if (dead) return;
    const float* ms = a.mscore + (size_t)hidx * a.T;
    const uint16_t* valid = a.valid + (size_t)b * a.T;
    const int i0 = (wi * 32 + lane) * KPT;
    uint32_t key[KPT], hi = 0u, lo = 0xffffffffu;
#pragma unroll
    for (int j = 0; j < KPT; j += 4) {
        if ((a.T & 3) == 0 && i0 + j + 4 <= Tv) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(ms + i0 + j));
            key[j] = sentry_order_key(v.x); key[j + 1] = sentry_order_key(v.y);
            key[j + 2] = sentry_order_key(v.z); key[j + 3] = sentry_order_key(v.w);
        } else {
#pragma unroll
            for (int e = j; e < j + 4; ++e) key[e] = i0 + e < Tv ? sentry_order_key(__ldg(ms + i0 + e)) : 0u;
        }
    }
#pragma unroll
    for (int j = 0; j < KPT; ++j)
        if (i0 + j < Tv) { hi = max(hi, key[j]); lo = min(lo, key[j]); }
    HeadReduce<NW> R{s_x, 0, lane, warp};
    R.max_min(hi, lo);
    uint32_t t = lo;
    bool cut = Tv == U;            // exactly U keys are >= t
#pragma unroll 1
    for (bool settled = false; !cut; settled = true) {
        int bit = hi != lo ? (31 - __clz((int)(hi ^ lo))) | 1 : -1;   // digits of two bits, aligned
        t = bit < 0 ? lo : (bit == 31 ? 0u : hi & ~((2u << bit) - 1u));
#pragma unroll 1
        for (bit -= 1; bit >= 0 && !cut; bit -= 2) {
            const uint32_t c1 = t + (1u << bit), c2 = t + (2u << bit), c3 = t + (3u << bit);
            uint32_t n12 = 0u, n3 = 0u;                    // counts above c1 (low half), c2 (high half) and c3
#pragma unroll
            for (int j = 0; j < KPT; ++j) {
                n12 += (key[j] >= c1 ? 1u : 0u) + (key[j] >= c2 ? 65536u : 0u);
                n3 += key[j] >= c3 ? 1u : 0u;
            }
            R.sum3(n12, n3);
            const int k1 = (int)(n12 & 0xffffu), k2 = (int)(n12 >> 16), k3 = (int)n3;
            if (k3 >= U) { t = c3; cut = k3 == U; }
            else if (k2 >= U) { t = c2; cut = k2 == U; }
            else if (k1 >= U) { t = c1; cut = k1 == U; }
        }
        if (settled) break;        // (not cut: ties of exact keys at t)
        uint32_t u = 0u, m = 0xffffffffu;   // the largest key not kept, the U-th key (ties: the same)
#pragma unroll
        for (int j = 0; j < KPT; ++j) {
            if (i0 + j >= Tv) continue;
            if (key[j] >= t) m = min(m, key[j]);
            else u = max(u, key[j]);
        }
        R.max_min(u, m);
        const bool finite = lo > 0x007fffffu && hi < 0xff800000u;
        uint32_t k_up = 0xffffffffu, k_dn = 0u;            // NaN or infinite scores: everything is contested
        if (finite) {
            const float margin = 2.0f * kScoreMargin * fmaxf(fabsf(order_key_value(hi)), fabsf(order_key_value(lo)));
            if (cut && order_key_value(m) - order_key_value(u) > margin) break;
            k_up = sentry_order_key(order_key_value(m) + margin);
            k_dn = sentry_order_key(order_key_value(m) - margin);
        }
        // surely active entries get the top key, hopeless ones zero, contested ones their exact key
        const uint32_t mask = a.masks[b];
        SampleSrc src;
        src.score_mode = a.score_mode;
        src.n_s = U;
        src.cnt = a.score_mode != 1 ? U : Tv;
        src.tbl = nullptr;
        if (a.score_mode != 1 && mask < (uint32_t)a.n_subsets && a.offsets[mask] >= 0) src.tbl = a.table + a.offsets[mask];
        const bool scored = src.tbl != nullptr || a.score_mode == 1;
        const __nv_bfloat16* qh = a.Q + ((size_t)b * a.Hq + h) * a.T * D;
        const __nv_bfloat16* Kg = a.K + ((size_t)b * a.Hk + h / (a.Hq / a.Hk)) * a.T * D;
#pragma unroll
        for (int j = 0; j < KPT; ++j) {
            const bool in = i0 + j < Tv, open = in && key[j] >= k_dn && key[j] <= k_up;
            unsigned todo = __ballot_sync(0xffffffffu, open);
            uint32_t nk = in && key[j] > k_up ? 0xffffffffu : 0u;
            while (todo) {
                const int sl = __ffs(todo) - 1;
                todo &= todo - 1;
                const int p = (wi * 32 + sl) * KPT + j;
                const uint32_t e = scored ? exact_score_key<D>(qh + (size_t)valid[p] * D, Kg, valid, Tv, src, p) : 1u;
                if (lane == sl) nk = min(max(e, 1u), 0xfffffffeu);
            }
            key[j] = nk;
        }
        hi = 0xffffffffu;
        lo = 0u;
        cut = false;
    }
    // ordered compaction: everything above t and, in index order, as many of the entries equal to t as are wanted
    uint32_t mine = 0u;            // above t: low half, equal to t: high half
#pragma unroll
    for (int j = 0; j < KPT; ++j)
        if (i0 + j < Tv) mine += (key[j] > t ? 1u : 0u) + (key[j] == t ? 65536u : 0u);
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    uint32_t before = incl - mine, total = __shfl_sync(0xffffffffu, incl, 31);
    if constexpr (NW > 1) {
        __syncthreads();
        if (lane == 0) s_x[0][2][warp] = total;
        __syncthreads();
        total = 0u;
#pragma unroll
        for (int w = 0; w < NW; ++w) { if (w == warp) before += total; total += s_x[0][2][w]; }
    }
    const int need_eq = cut ? 0x7fffffff : U - (int)(total & 0xffffu);
    int gt_n = (int)(before & 0xffffu), eq_n = (int)(before >> 16);
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
        const bool in = i0 + j < Tv, is_gt = in && key[j] > t, is_eq = in && key[j] == t;
        if (is_gt || (is_eq && eq_n < need_eq)) out[gt_n + min(eq_n, need_eq)] = (int32_t)valid[i0 + j];
        gt_n += is_gt;
        eq_n += is_eq;
    }
}

// ------------------------------------------------------------------------------------------ rows
// D/4 consecutive output elements of a row (the columns a lane owns: see below), rounded and stored.
template <int D>
__device__ __forceinline__ void store_cols(__nv_bfloat16* dst, const float (&acc)[D / 8][4], int h2, float inv) {
    constexpr int NT = D / 8;
    uint32_t w[NT];
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        // element e of the lane's D/4: tile e % NT, accumulator column e / NT
        const int e0 = 2 * i, e1 = 2 * i + 1;
        w[i] = pack2(acc[e0 % NT][2 * h2 + e0 / NT] * inv, acc[e1 % NT][2 * h2 + e1 / NT] * inv);
    }
    if constexpr (D == 16) {
        *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
    } else {
#pragma unroll
        for (int i = 0; i < NT / 4; ++i)
            reinterpret_cast<uint4*>(dst)[i] = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
    }
}
__host__ __device__ constexpr int part_words(int D) { return D / 2 + 4; }   // accumulator, maxima and sums of a lane

// What a block needs to know of its group: heads (shared), T_v, active rows per head.
struct GroupInfo { int b, g, Tv, rk, Ue, n_tiles; };
__device__ __forceinline__ GroupInfo group_info(const SplitArgs& a, int grp, int* s_hs, int* s_khs, int* s_rk) {
    GroupInfo q;
    q.b = grp / a.Hk;
    q.g = grp % a.Hk;
    if (threadIdx.x < 32) {
        bool bad;
        const int n = warp_group_heads(a.kept_heads + (size_t)q.b * a.k_h, a.k_h, a.Hq / a.Hk, q.g, a.Hq, s_hs, s_khs, bad);
        if (threadIdx.x == 0) *s_rk = n;
    }
    q.Tv = a.tv[q.b];
    __syncthreads();
    q.rk = *s_rk;
    q.Ue = a.given ? a.U_max : sentry_num_active(q.Tv, a.c);
    q.n_tiles = (q.rk * q.Ue + 15) / 16;
    return q;
}
// Token of active row r (heads packed back to back) or -1; kh: its kept-list slot, h: its head.
__device__ __forceinline__ int active_token(const SplitArgs& a, const GroupInfo& q, const int* s_hs, const int* s_khs, int r,
                                            uint32_t mask, int& h, int& kh) {
    h = s_hs[0];
    kh = s_khs[0];
    if (r >= q.rk * q.Ue) return -1;
    const int hh = r / q.Ue;
    h = s_hs[hh];
    kh = s_khs[hh];
    int t = a.active[((size_t)q.b * a.k_h + kh) * a.U_max + r - hh * q.Ue];
    if (a.given && t >= 0) {       // the caller's rows: only present tokens count
        const int m = t < a.T ? a.ids[t] : -1;
        if (!(m >= 0 && m < 32 && ((mask >> m) & 1u))) { atomicOr(a.status, SENTRY_STATUS_BIT_BAD_INDEX); t = -1; }
    }
    return t;
}

// grid B * Hk * nsplit.  A warp takes a tile of 16 active rows (of any of the group's heads: they share K and V) over this
// block's part of the keys; online softmax, every weight as a 16-bit head plus a 16-bit remainder (p = p_hi + p_lo to
// 2^-17, so the rounding of the weights drops out of O).  K and V fragments come straight from global memory (L1 serves
// the tiles of a block from one fetch): 16 bytes of a key row per lane for Q K^T, and for P V the dims are numbered so that
// a lane holds D/8 consecutive ones of four keys, which two byte permutations turn into operand pairs; the accumulator
// columns a lane then owns are D/4 consecutive dims.  Bound by the warp MMA (24 of them per 16 rows x 32 keys at d = 32).
template <int D>
__global__ void __launch_bounds__(kSplitThreads, 2)
attend_split_rows_kernel(const __grid_constant__ SplitArgs a) {
    constexpr int NT = D / 8, KS = D / 16, W = D / 8;
    extern __shared__ __align__(128) uint8_t s_raw[];
    __shared__ int s_hs[kMaxRK], s_khs[kMaxRK], s_rk;
    uint16_t* s_tok = reinterpret_cast<uint16_t*>(s_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gq = lane >> 2, tq = lane & 3;
    const int grp = blockIdx.x / a.nsplit, sp = blockIdx.x % a.nsplit;
    grid_dependency_wait();
    const GroupInfo q = group_info(a, grp, s_hs, s_khs, &s_rk);
    if (q.rk == 0 || q.Tv == 0) return;
    const int n32 = (q.Tv + 31) / 32, k0 = sp * n32 / a.nsplit * 32, k1 = min(q.Tv, (sp + 1) * n32 / a.nsplit * 32);
    const int n_keys = k1 - k0;    // may be 0: the part is then empty (sum 0)
    for (int i = threadIdx.x; i < n_keys; i += kSplitThreads) s_tok[i] = a.valid[(size_t)q.b * a.T + k0 + i];
    __syncthreads();
    const uint32_t mask = a.masks[q.b];
    const __nv_bfloat16* Kg = a.K + (size_t)grp * a.T * D;
    const __nv_bfloat16* Vg = a.V + (size_t)grp * a.T * D + gq * (D / 8);
    const float sl2 = rsqrtf((float)D) * 1.4426950408889634f;  // scale * log2(e)
    for (int tile = warp; tile < q.n_tiles; tile += kSplitWarps) {
        uint32_t qf[2][W];
        int tok[2], kh[2];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            int h;
            tok[half] = active_token(a, q, s_hs, s_khs, tile * 16 + gq + half * 8, mask, h, kh[half]);
#pragma unroll
            for (int i = 0; i < W; ++i) qf[half][i] = 0u;
            if (tok[half] >= 0) ld_row_frag<D>(qf[half], a.Q + (((size_t)q.b * a.Hq + h) * a.T + tok[half]) * D, tq);
        }
        float acc[NT][4], m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
#pragma unroll 1
        for (int kk = 0; kk < n_keys; kk += 32) {
            // V of keys 2 tq, 2 tq + 1 and the two 8 further on (both halves of the step), dims gq * D/8 ..: on the way while
            // the scores and their softmax are computed
            uint32_t v[2][4][NT / 2];
#pragma unroll
            for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int key = min(kk + ks * 16 + 2 * tq + (i & 1) + (i >> 1) * 8, n_keys - 1);
                    const __nv_bfloat16* src = Vg + (uint32_t)s_tok[key] * D;
                    if constexpr (D == 16) {
                        v[ks][i][0] = __ldg(reinterpret_cast<const uint32_t*>(src));
                    } else if constexpr (D == 32) {
                        const uint2 x = __ldg(reinterpret_cast<const uint2*>(src));
                        v[ks][i][0] = x.x; v[ks][i][1] = x.y;
                    } else {
                        const uint4 x = __ldg(reinterpret_cast<const uint4*>(src));
                        v[ks][i][0] = x.x; v[ks][i][1] = x.y; v[ks][i][2] = x.z; v[ks][i][3] = x.w;
                    }
                }
            float s[4][4];
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                uint32_t kf[W];
                ld_row_frag<D>(kf, Kg + (uint32_t)s_tok[min(kk + nt * 8 + gq, n_keys - 1)] * D, tq);
#pragma unroll
                for (int e = 0; e < 4; ++e) s[nt][e] = 0.f;
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) {
                    const uint32_t af[4] = {qf[0][2 * ks], qf[1][2 * ks], qf[0][2 * ks + 1], qf[1][2 * ks + 1]};
                    mma_bf16_16816(s[nt], af, kf[2 * ks], kf[2 * ks + 1]);
                }
            }
            if (kk + 32 > n_keys) {   // the last, partial step: keys past the end drop out
#pragma unroll
                for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (kk + nt * 8 + tq * 2 + (e & 1) >= n_keys) s[nt][e] = -INFINITY;
            }
            float mt[2] = {-INFINITY, -INFINITY}, corr[2], ms[2];
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                mt[0] = max3(mt[0], s[nt][0], s[nt][1]);
                mt[1] = max3(mt[1], s[nt][2], s[nt][3]);
            }
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) {
                mt[h2] = fmaxf(mt[h2], __shfl_xor_sync(0xffffffffu, mt[h2], 1));
                mt[h2] = fmaxf(mt[h2], __shfl_xor_sync(0xffffffffu, mt[h2], 2));
                const float m_new = fmaxf(m_run[h2], mt[h2]);
                corr[h2] = fast_exp2((m_run[h2] - m_new) * sl2);   // 0 on the first step
                m_run[h2] = m_new;
                ms[h2] = m_new * sl2;
                l_run[h2] *= corr[h2];
            }
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) s[nt][e] = fast_exp2(fmaf(s[nt][e], sl2, -ms[e >> 1]));
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                acc[n][0] *= corr[0]; acc[n][1] *= corr[0];
                acc[n][2] *= corr[1]; acc[n][3] *= corr[1];
            }
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
                uint32_t pa[4], pb[4];
                pa[0] = pack2(s[2 * ks][0], s[2 * ks][1]);
                pa[1] = pack2(s[2 * ks][2], s[2 * ks][3]);
                pa[2] = pack2(s[2 * ks + 1][0], s[2 * ks + 1][1]);
                pa[3] = pack2(s[2 * ks + 1][2], s[2 * ks + 1][3]);
                pb[0] = pack2_rem(s[2 * ks][0], s[2 * ks][1], pa[0]);
                pb[1] = pack2_rem(s[2 * ks][2], s[2 * ks][3], pa[1]);
                pb[2] = pack2_rem(s[2 * ks + 1][0], s[2 * ks + 1][1], pa[2]);
                pb[3] = pack2_rem(s[2 * ks + 1][2], s[2 * ks + 1][3], pa[3]);
                l_run[0] += (s[2 * ks][0] + s[2 * ks][1]) + (s[2 * ks + 1][0] + s[2 * ks + 1][1]);
                l_run[1] += (s[2 * ks][2] + s[2 * ks][3]) + (s[2 * ks + 1][2] + s[2 * ks + 1][3]);
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const uint32_t sel = (j & 1) ? 0x7632u : 0x5410u;
                    const uint32_t b0 = __byte_perm(v[ks][0][j / 2], v[ks][1][j / 2], sel),
                                   b1 = __byte_perm(v[ks][2][j / 2], v[ks][3][j / 2], sel);
                    mma_bf16_16816(acc[j], pa, b0, b1);
                    mma_bf16_16816(acc[j], pb, b0, b1);
                }
            }
        }
        if (a.nsplit == 1) {
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) {
                float l = l_run[h2];
                l += __shfl_xor_sync(0xffffffffu, l, 1);
                l += __shfl_xor_sync(0xffffffffu, l, 2);
                if (tok[h2] >= 0)
                    store_cols<D>(a.O + (((size_t)q.b * a.k_h + kh[h2]) * a.T + tok[h2]) * D + tq * (D / 4), acc, h2, 1.0f / l);
            }
        } else {
            float* dst = a.part + (((size_t)grp * a.nsplit + sp) * kRowTiles + tile) * part_words(D) * 32 + lane;
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) dst[(n * 4 + e) * 32] = acc[n][e];
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) { dst[(NT * 4 + h2) * 32] = m_run[h2]; dst[(NT * 4 + 2 + h2) * 32] = l_run[h2]; }
        }
    }
}

// ------------------------------------------------------------------------------------------ fill
// grid (B * Hk, token slices).  Context rows (mean of V_g) on the present tokens that are not active, zeros on absent
// ones, 16 bytes per store; with the keys in parts, the slices also share out the row tiles and merge their parts.
// Bound by writing O.
// P: room for the parts (1: none to merge).  16 parts of loads in flight take 80 registers, 3 blocks per SM; fewer parts
// leave more.
template <int D, int P>
__global__ void __launch_bounds__(kSplitThreads, P < 16 ? 4 : (D == 64 ? 2 : 3))
attend_split_fill_kernel(const __grid_constant__ SplitArgs a) {
    constexpr int NT = D / 8, CPR = D / 8;
    extern __shared__ __align__(128) uint8_t s_raw[];   // active bits [kMaxRK][words of the slice]
    __shared__ int s_hs[kMaxRK], s_khs[kMaxRK], s_rk;
    __shared__ __align__(16) unsigned short s_mean[D];
    __shared__ float s_acc[P > 1 ? D / 2 : 1][32];
    uint32_t* s_bits = reinterpret_cast<uint32_t*>(s_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gq = lane >> 2, tq = lane & 3;
    const int grp = blockIdx.x;
    const int per = ((a.T + (int)gridDim.y - 1) / (int)gridDim.y + 31) & ~31;
    const int t0 = (int)blockIdx.y * per, t1 = min(a.T, t0 + per), words = per / 32;
    for (int i = threadIdx.x; i < kMaxRK * words; i += kSplitThreads) s_bits[i] = 0u;
    grid_dependency_wait();
    const GroupInfo q = group_info(a, grp, s_hs, s_khs, &s_rk);
    if (q.rk == 0) return;
    const uint32_t mask = a.masks[q.b];
    if (q.Tv > 0) {
        if (threadIdx.x < D) {
            const int nb = (q.Tv + kScoreBlock - 1) / kScoreBlock;
            const float* vs = a.vsum + (size_t)grp * a.n_blk * D + threadIdx.x;
            float t = 0.f;
            for (int i0 = 0; i0 < nb; i0 += 16) {   // 16 sums on the way at once, added in order
                float v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = i0 + i < nb ? vs[(i0 + i) * D] : 0.f;
#pragma unroll
                for (int i = 0; i < 16; ++i) t += v[i];
            }
            s_mean[threadIdx.x] = att_bits(t / (float)q.Tv);
        }
        for (int r = threadIdx.x; r < q.rk * q.Ue; r += kSplitThreads) {
            int h, kh;
            const int t = active_token(a, q, s_hs, s_khs, r, mask, h, kh);
            if (t >= t0 && t < t1) atomicOr(&s_bits[r / q.Ue * words + ((t - t0) >> 5)], 1u << ((t - t0) & 31));
        }
    }
    __syncthreads();
    if constexpr (P > 1) if (q.Tv > 0) {
        // the parts of a row tile, by the whole block: a warp takes D/16 of the lanes' D/2 accumulator words, and all loads of
        // all parts are on the way at once (one warp per tile, part after part, took 40 of the launch's 48 K cycles)
        const float sl2 = rsqrtf((float)D) * 1.4426950408889634f;
        const size_t step = (size_t)kRowTiles * part_words(D) * 32;
        for (int tile = (int)blockIdx.y; tile < q.n_tiles; tile += (int)gridDim.y) {
            const float* src = a.part + ((size_t)grp * a.nsplit * kRowTiles + tile) * part_words(D) * 32 + lane;
            float w[2][P], v[D / 16][P];
#pragma unroll
            for (int sp = 0; sp < P; ++sp) {
                const bool in = sp < a.nsplit;
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2) w[h2][sp] = in ? src[sp * step + (NT * 4 + h2) * 32] : -INFINITY;
#pragma unroll
                for (int k = 0; k < D / 16; ++k) v[k][sp] = in ? src[sp * step + (warp * (D / 16) + k) * 32] : 0.f;
            }
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) {
                float m = w[h2][0];
#pragma unroll
                for (int sp = 1; sp < P; ++sp) m = fmaxf(m, w[h2][sp]);
#pragma unroll
                for (int sp = 0; sp < P; ++sp)
                    w[h2][sp] = w[h2][sp] == -INFINITY ? 0.f : fast_exp2((w[h2][sp] - m) * sl2);   // (empty parts: 0)
            }
#pragma unroll
            for (int k = 0; k < D / 16; ++k) {
                const int h2 = ((warp * (D / 16) + k) >> 1) & 1;
                float t = 0.f;
#pragma unroll
                for (int sp = 0; sp < P; ++sp) t = fmaf(v[k][sp], h2 ? w[1][sp] : w[0][sp], t);
                s_acc[warp * (D / 16) + k][lane] = t;
            }
            __syncthreads();
            if (warp < 2) {   // warp h2: rows gq + 8 h2 of the tile
                float l = 0.f, acc[NT][4];
#pragma unroll
                for (int sp = 0; sp < P; ++sp)
                    if (sp < a.nsplit) l = fmaf(src[sp * step + (NT * 4 + 2 + warp) * 32], warp ? w[1][sp] : w[0][sp], l);
                l += __shfl_xor_sync(0xffffffffu, l, 1);
                l += __shfl_xor_sync(0xffffffffu, l, 2);
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int e = 0; e < 2; ++e) acc[n][e] = s_acc[n * 4 + 2 * warp + e][lane];
                int h, kh;
                const int t = active_token(a, q, s_hs, s_khs, tile * 16 + gq + warp * 8, mask, h, kh);
                if (t >= 0) store_cols<D>(a.O + (((size_t)q.b * a.k_h + kh) * a.T + t) * D + tq * (D / 4), acc, 0, 1.0f / l);
            }
            __syncthreads();
        }
    }
    const uint4* mean4 = reinterpret_cast<const uint4*>(s_mean);
    for (int hh = 0; hh < q.rk; ++hh) {
        uint4* dst = reinterpret_cast<uint4*>(a.O + ((size_t)q.b * a.k_h + s_khs[hh]) * a.T * D);
        const uint32_t* bits = s_bits + hh * words;
#pragma unroll 4
        for (int i = t0 * CPR + threadIdx.x; i < t1 * CPR; i += kSplitThreads) {
            const int t = i / CPR, cc = i % CPR;
            if ((bits[(t - t0) >> 5] >> ((t - t0) & 31)) & 1u) continue;
            const int m = __ldg(a.ids + t);
            dst[i] = m >= 0 && m < 32 && ((mask >> m) & 1u) ? mean4[cc] : make_uint4(0, 0, 0, 0);
        }
    }
}

// ------------------------------------------------------------------------------------------ launch
// Parts of the keys in the rows launch: about three blocks per SM, at least 256 keys a part, at most 16 parts.
int split_parts(const sentry_attend_desc& d) {
    const long long groups = (long long)d.B * d.Hk;
    long long n = (444 + groups - 1) / groups;
    const long long most = (d.T + 255) / 256;
    if (n > most) n = most;
    return (int)(n > kMaxParts ? kMaxParts : (n < 1 ? 1 : n));
}

struct SplitWs { uint16_t* valid; int* tv; float *vsum, *part; };
SplitWs split_carve(const sentry_attend_desc& d, WsAlloc& w) {
    const size_t groups = (size_t)d.B * d.Hk, n_blk = (size_t)(d.T + kScoreBlock - 1) / kScoreBlock;
    const int ns = split_parts(d);
    SplitWs s;
    s.valid = w.take<uint16_t>((size_t)d.B * d.T);
    s.tv = w.take<int>(d.B);
    s.vsum = w.take<float>(groups * n_blk * d.d);
    s.part = w.take<float>(ns > 1 ? groups * ns * kRowTiles * part_words(d.d) * 32 : 0);
    return s;
}

template <int D>
int launch_select(sentry_ctx* ctx, const SplitArgs& p, cudaStream_t st) {
    const unsigned heads = (unsigned)p.B * p.k_h, packs = (heads + kSplitWarps - 1) / kSplitWarps;
    LaunchScope ls(ctx, KS_ATT_SELECT, st);
#define SELECT(KPT, NW, GRID) SENTRY_CUDA_TRY(launch_chained(attend_split_select_kernel<D, KPT, NW>, dim3(GRID), dim3(kSplitThreads), 0, st, p))
    // a warp per head where there are enough heads to fill the GPU that way, or the list is short anyway
    if (p.T <= 256) SELECT(8, 1, packs);
    else if (p.T <= 512 && packs >= 64) SELECT(16, 1, packs);
    else if (p.T <= 1024 && packs >= 128) SELECT(32, 1, packs);
    else if (p.T <= 1024) SELECT(4, 8, heads);
    else if (p.T <= 2048) SELECT(8, 8, heads);
    else if (p.T <= 4096) SELECT(16, 8, heads);
    else SELECT(32, 8, heads);
#undef SELECT
    return SENTRY_OK;
}

template <int D>
int launch_d(sentry_ctx* ctx, const AttendArgs& a, const SplitWs& w, cudaStream_t st) {
    const sentry_attend_desc& d = a.d;
    SplitArgs p = {};
    p.Q = (const __nv_bfloat16*)a.Q; p.K = (const __nv_bfloat16*)a.K; p.V = (const __nv_bfloat16*)a.V;
    p.kept_heads = a.kept_heads; p.ids = a.ids; p.masks = a.masks;
    p.table = a.sample_table; p.offsets = a.sample_offsets; p.n_subsets = a.n_subsets;
    p.B = d.B; p.T = d.T; p.Hq = d.Hq; p.Hk = d.Hk; p.k_h = d.k_h; p.c = d.c; p.score_mode = d.score_mode; p.U_max = a.U_max;
    p.nsplit = split_parts(d);
    p.n_blk = (d.T + kScoreBlock - 1) / kScoreBlock;
    p.given = a.selection_given;
    p.gate_scores = a.gate_scores; p.gate_S = a.gate_S; p.kept_out = a.kept_out;
    p.mscore = a.mscore; p.valid = w.valid; p.tv = w.tv; p.vsum = w.vsum; p.part = w.part;
    p.active = a.active;
    p.O = (__nv_bfloat16*)a.O; p.status = a.status;
    const unsigned groups = (unsigned)d.B * d.Hk;
    const size_t list = (size_t)((d.T + 63) & ~63) * 2;
    {
        LaunchScope ls(ctx, KS_ATT_SCORE, st);
        SENTRY_CUDA_TRY(launch_chained(attend_split_score_kernel<D>, dim3(groups * (unsigned)p.n_blk), dim3(kSplitThreads),
                                       list + (size_t)kSplitWarps * 8 * kMaxActive * 2, st, p));
    }
    if (!p.given) {
        const int rc = launch_select<D>(ctx, p, st);
        if (rc != SENTRY_OK) return rc;
    }
    LaunchScope ls(ctx, KS_ATT_CORE, st, 2);
    SENTRY_CUDA_TRY(launch_chained(attend_split_rows_kernel<D>, dim3(groups * (unsigned)p.nsplit), dim3(kSplitThreads),
                                   list / p.nsplit + 128, st, p));
    // slices of the tokens: three or four blocks per SM, at least 64 tokens each
    long long slices = ((p.nsplit > 4 ? 3LL : 4LL) * ctx->sm_count + groups - 1) / groups;
    if (slices > (d.T + 63) / 64) slices = (d.T + 63) / 64;
    if (slices < 1) slices = 1;
    const size_t bits = (size_t)kMaxRK * (((d.T + slices - 1) / slices + 31) / 32) * 4;
    auto fill = p.nsplit == 1 ? attend_split_fill_kernel<D, 1> : (p.nsplit <= 4 ? attend_split_fill_kernel<D, 4> : attend_split_fill_kernel<D, kMaxParts>);
    SENTRY_CUDA_TRY(launch_chained(fill, dim3(groups, (unsigned)slices), dim3(kSplitThreads), bits, st, p));
    return SENTRY_OK;
}

}  // namespace

size_t attend_split_ws_bytes(const sentry_attend_desc& d) {
    WsAlloc a(nullptr, 0);
    (void)split_carve(d, a);
    return a.off + 256;
}

int launch_attend_split(sentry_ctx* ctx, const AttendArgs& a, WsAlloc& ws, cudaStream_t st) {
    const SplitWs w = split_carve(a.d, ws);
    if (!ws.ok) return SENTRY_ERR_WORKSPACE;
    switch (a.d.d) {
        case 16: return launch_d<16>(ctx, a, w, st);
        case 32: return launch_d<32>(ctx, a, w, st);
        case 64: return launch_d<64>(ctx, a, w, st);
        default: return SENTRY_ERR_UNSUPPORTED;
    }
}
