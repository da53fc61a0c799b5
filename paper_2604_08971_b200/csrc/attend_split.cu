// SentryAttend (Section 4.4, Eq. 6) for 16-bit tensors in four launches, each of which spreads over the whole GPU:
//
//   score   a warp scores batches of 8 query positions of one (sample, KV group) for all kept heads, with the arithmetic of
//           the one-launch form (fused_score_pass), the sampled key rows copied to shared memory a few steps ahead; the
//           block also lists the sample's present tokens and sums V over its positions
//   select  the U best positions per head, a warp (T <= 1024) or a block each
//   rows    Eq. 6 on tiles of 16 active rows, a warp per tile and part of the keys, K and V fragments from global memory
//   fill    context and zero rows, and the merge of the key parts
//
// A CTA per (sample, group) does the same in attend_bf16.cu and attend_long.cu: ten phases with a barrier after each, of
// which every one is a chain of latencies, on as many SMs as there are groups.  Taken apart, each phase runs with as many
// warps as it has work: the form for long sequences and for few groups (attend_split_faster in api.cu has the line).
// Measured on 16 x 4096 tokens, d = 32, 4 of 8 heads kept, one to three of three modalities present: 310 us in one CTA per
// group, 80 as four launches.
#include <math.h>
#include <stddef.h>

#include <type_traits>

#include "attend_common.cuh"

namespace {

constexpr int kSplitThreads = 256, kSplitWarps = kSplitThreads / 32;
constexpr int kScoreBlock = 128;                 // query positions per score block (or two blocks with half of them each)
constexpr int kRowTiles = kMaxRK * kMaxActive / 16;
constexpr int kMaxParts = 16;                     // parts of the keys in the rows launch

// ------------------------------------------------------------------------------------------ pieces
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

// Present-token list of a sample, ascending, by 256 threads: every warp a run of 128-token pieces, four tokens to a lane and
// all its loads on the way at once.  red: kSplitWarps ints.  Returns T_v; the list is complete behind the caller's next
// barrier -- where T_v is above needed_from: there is nothing to do with the list otherwise.
__device__ __forceinline__ int list_present(const int32_t* __restrict__ ids, int T, uint32_t mask, uint16_t* valid, int* red,
                                            int needed_from) {
    constexpr int MOST = 8192 / (128 * kSplitWarps);   // pieces of a warp's run (attend_bf16_supported: T <= 8192)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = ((T + 127) / 128 + kSplitWarps - 1) / kSplitWarps, t0 = warp * per * 128 + lane * 4;
    const bool wide = ((uintptr_t)ids & 15) == 0;
    int4 id[MOST];
#pragma unroll
    for (int j = 0; j < MOST; ++j) {
        const int t = t0 + j * 128;
        id[j] = make_int4(-1, -1, -1, -1);
        if (j >= per || t >= T) continue;
        if (wide && t + 4 <= T) {
            id[j] = __ldg(reinterpret_cast<const int4*>(ids + t));
        } else {
            id[j].x = __ldg(ids + t);
            if (t + 1 < T) id[j].y = __ldg(ids + t + 1);
            if (t + 2 < T) id[j].z = __ldg(ids + t + 2);
            if (t + 3 < T) id[j].w = __ldg(ids + t + 3);
        }
    }
    auto present = [&](int m) { return m >= 0 && m < 32 ? (mask >> m) & 1u : 0u; };
    uint32_t bits = 0u;                            // four per piece
#pragma unroll
    for (int j = 0; j < MOST; ++j)
        bits |= (present(id[j].x) | present(id[j].y) << 1 | present(id[j].z) << 2 | present(id[j].w) << 3) << (4 * j);
    const int mine = __reduce_add_sync(0xffffffffu, __popc(bits));
    if (lane == 0) red[warp] = mine;
    __syncthreads();
    int base = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kSplitWarps; ++w) { const int c = red[w]; total += c; if (w < warp) base += c; }
    if (total <= needed_from) return total;
#pragma unroll
    for (int j = 0; j < MOST; ++j) {
        if (j >= per) break;
        const uint32_t b4 = bits >> (4 * j) & 15u, lt = (1u << lane) - 1u;
        int at = base;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t bm = __ballot_sync(0xffffffffu, (b4 >> k) & 1u);
            at += __popc(bm & lt);
            base += __popc(bm);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if ((b4 >> k) & 1u) valid[at++] = (uint16_t)(t0 + j * 128 + k);
    }
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
// A warp scores batches of 8 query positions; the four lanes of a quad take four keys of one of them.  Shared memory of a
// block: per warp a ring of copied key rows (a step's 32, one per lane) and the tokens of its batches' sampled keys, then
// the sample's present-token list.
constexpr int kBatch = 8;                         // query positions of a batch
constexpr int kBatches = kScoreBlock / (kBatch * kSplitWarps);   // of a warp
constexpr int kBatchSteps = kMaxActive / 4;       // steps of a batch: a key for each lane of a quad
template <int D>
struct ScoreSmem {
    static constexpr int STAGES = D == 64 ? 2 : 3;   // two blocks fit an SM at every T
    static constexpr int STAGE_BYTES = 32 * D * 2;
    static constexpr int RING_BYTES = STAGES * STAGE_BYTES;
    static constexpr int TOK_AT = kSplitWarps * RING_BYTES;
    static constexpr int VALID_AT = TOK_AT + kSplitWarps * kBatches * kBatchSteps * 32 * 2;
};

// Tokens of the sampled keys of a warp's batches, 32 per step.  Row r = 4 q + a of a step (query q, key a of its four) is at
// (r % RPC) CPR + r / RPC: the CPR tokens that a lane copies chunks of are then one word of shared memory.  Positions outside
// the list are flagged and count as position 0; keys from n_s on (to a multiple of 4) repeat the last one, queries past the
// list those of the last.
template <int CPR>
__device__ __forceinline__ void stage_tokens(const int32_t* __restrict__ tbl, int score_mode, int n_s, int p0, int batches, int Tv,
                                             const uint16_t* s_valid, uint16_t* s_tok, unsigned int* status) {
    constexpr int RPC = 32 / CPR;
    const int lane = threadIdx.x & 31, q = lane & 7, a4 = lane >> 3, n4 = (n_s + 3) & ~3, r = 4 * q + a4;
    const size_t es = score_mode == 2 ? (size_t)Tv : 1;
    int e[kBatches][kBatchSteps];                  // all of a lane's table entries on the way at once
#pragma unroll
    for (int b = 0; b < kBatches; ++b) {
        const int p = min(p0 + b * kBatch * kSplitWarps + q, Tv - 1);
        const int32_t* src = tbl + (score_mode == 2 ? (size_t)p : (size_t)p * n_s);
#pragma unroll
        for (int i = 0; i < kBatchSteps; ++i)
            e[b][i] = b < batches && 4 * i < n4 ? __ldg(src + (size_t)min(4 * i + a4, n_s - 1) * es) : 0;
    }
    bool bad = false;
#pragma unroll
    for (int b = 0; b < kBatches; ++b) {
        if (b >= batches) break;
#pragma unroll
        for (int i = 0; i < kBatchSteps; ++i) {
            if (4 * i >= n4) break;
            if ((unsigned)e[b][i] >= (unsigned)Tv) { bad = true; e[b][i] = 0; }
            s_tok[(b * kBatchSteps + i) * 32 + r % RPC * CPR + r / RPC] = s_valid[e[b][i]];
        }
    }
    if (bad) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
}
// N tokens from shared memory in one load.
template <int N>
__device__ __forceinline__ void load_tokens(uint32_t (&t)[N], const uint16_t* s) {
    uint32_t w[N / 2];
    if constexpr (N == 2) {
        w[0] = *reinterpret_cast<const uint32_t*>(s);
    } else if constexpr (N == 4) {
        const uint2 v = *reinterpret_cast<const uint2*>(s);
        w[0] = v.x; w[1] = v.y;
    } else {
        const uint4 v = *reinterpret_cast<const uint4*>(s);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    }
#pragma unroll
    for (int i = 0; i < N; ++i) t[i] = (i & 1) ? w[i / 2] >> 16 : w[i / 2] & 0xffffu;
}

// The query rows of a token, as they are stored.
template <int D, int NH>
__device__ __forceinline__ void load_queries(uint32_t (&q)[NH][D / 2], const __nv_bfloat16* const (&qh)[NH], uint32_t tok) {
#pragma unroll
    for (int h = 0; h < NH; ++h)
#pragma unroll
        for (int c = 0; c < D / 8; ++c) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(qh[h] + tok * D) + c);
            q[h][4 * c] = v.x; q[h][4 * c + 1] = v.y; q[h][4 * c + 2] = v.z; q[h][4 * c + 3] = v.w;
        }
}
// Dot products of NH query rows with a key row, chunk by chunk (8 elements) from `chunk`, each in the four accumulators and
// the order of the one-launch form (fused_score_pass), so that the two forms round alike.
template <int D, int NH, typename Chunk>
__device__ __forceinline__ void dot_rows(const uint32_t (&q)[NH][D / 2], Chunk chunk, float scale, float (&sc)[NH]) {
    float acc[NH][4];
#pragma unroll
    for (int h = 0; h < NH; ++h) acc[h][0] = acc[h][1] = acc[h][2] = acc[h][3] = 0.f;
#pragma unroll
    for (int c = 0; c < D / 8; ++c) {
        const uint4 v = chunk(c);
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            fma_bf16_pair(acc[h][0], acc[h][1], q[h][4 * c], v.x);
            fma_bf16_pair(acc[h][2], acc[h][3], q[h][4 * c + 1], v.y);
            fma_bf16_pair(acc[h][0], acc[h][1], q[h][4 * c + 2], v.z);
            fma_bf16_pair(acc[h][2], acc[h][3], q[h][4 * c + 3], v.w);
        }
    }
#pragma unroll
    for (int h = 0; h < NH; ++h) sc[h] = __fmul_rn((acc[h][0] + acc[h][1]) + (acc[h][2] + acc[h][3]), scale);
}

// Scores M = max_j s_j - mean_j s_j of NH heads for the warp's batches of query positions (p: the quad's in the first one)
// over their sampled keys, in table order.  The rows come through the warp's ring, STAGES - 1 steps ahead, copied with D/8
// lanes to a row, so that a copy instruction touches few lines, and read back as a whole row per lane without bank
// conflicts (Sw).  Every lane of the quad adds the quad's four scores in key order.
template <int D, int NH>
__device__ __forceinline__ void score_sampled(const __nv_bfloat16* const (&qh)[NH], const __nv_bfloat16* __restrict__ Kg,
                                              float* const (&out)[NH], const uint16_t* s_valid, const uint16_t* s_tok,
                                              uint32_t ring, int n_s, int p, int batches, int Tv) {
    using S = Sw<D>;
    using M = ScoreSmem<D>;
    constexpr int RPC = 32 / S::CPR;                // rows of a copy instruction
    const int lane = threadIdx.x & 31, tq = lane & 3, row0 = lane / S::CPR, cc = lane % S::CPR;
    const float scale = rsqrtf((float)D), inv_cnt = 1.0f / (float)n_s;
    const int steps = (n_s + 3) / 4;                // of a batch
    const __nv_bfloat16* Kc = Kg + cc * 8;
    const uint32_t copy_to = ring + S::off(row0, cc), row_at = ring + S::off(lane, 0);
    const uint16_t* tp = s_tok + row0 * S::CPR;
    int f_left = batches * steps, f_step = 0;       // what is still to be fetched
    auto fetch = [&](uint32_t stage) {              // stage: byte offset in the ring
        if (f_left > 0) {
            uint32_t t[S::CPR];
            load_tokens(t, tp + f_step * 32);
#pragma unroll
            for (int i = 0; i < S::CPR; ++i) {
                // (row i * RPC + row0 is swizzled as row0 is; d = 64: with bit 2 of the row in every other i)
                const uint32_t to = (D == 64 ? copy_to ^ ((i & 1) << 6) : copy_to) + stage + i * RPC * S::RB;
                ptx::cp_async_16(to, Kc + t[i] * D);
            }
            --f_left;
            if (++f_step == steps) { f_step = 0; tp += kBatchSteps * 32; }
        }
        ptx::cp_async_commit();
    };
    __syncwarp();                                   // the ring is free, the tokens are there
#pragma unroll
    for (int s = 0; s < M::STAGES - 1; ++s) fetch(s * M::STAGE_BYTES);
    uint32_t stage = 0, ahead = M::RING_BYTES - M::STAGE_BYTES;
#pragma unroll 1
    for (int batch = 0; batch < batches; ++batch, p += kBatch * kSplitWarps) {
        uint32_t q[NH][D / 2];
        load_queries<D, NH>(q, qh, s_valid[min(p, Tv - 1)]);
        float mx[NH], sum[NH], sc[NH];
#pragma unroll
        for (int h = 0; h < NH; ++h) { mx[h] = -INFINITY; sum[h] = 0.f; }
        auto take = [&](int n) {                    // the quad's four scores, of which n count
#pragma unroll
            for (int h = 0; h < NH; ++h) {
                float v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) v[j] = __shfl_sync(0xffffffffu, sc[h], j, 4);
                if (n >= 4) {
                    mx[h] = fmaxf(mx[h], sc[h]);
                    sum[h] = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(sum[h], v[0]), v[1]), v[2]), v[3]);
                } else {
                    if (tq < n) mx[h] = fmaxf(mx[h], sc[h]);
#pragma unroll
                    for (int j = 0; j < 3; ++j)
                        if (j < n) sum[h] = __fadd_rn(sum[h], v[j]);
                }
            }
        };
#pragma unroll 1
        for (int step = 0; step < steps; ++step) {
            ptx::cp_async_wait_group<M::STAGES - 2>();
            __syncwarp();                           // every lane's copies of this step are there, the stage before is free
            const uint32_t addr = row_at + stage;
            constexpr int EARLY = S::CPR <= 4 ? S::CPR : 2;   // under way while the step before is taken in
            uint4 v[EARLY];
#pragma unroll
            for (int c = 0; c < EARLY; ++c) v[c] = lds128(addr ^ (c << 4));
            fetch(ahead);
            if (step > 0) take(4);
            dot_rows<D, NH>(q, [&](int c) { return c < EARLY ? v[c] : lds128(addr ^ (c << 4)); }, scale, sc);
            ahead = stage;
            stage = stage == M::RING_BYTES - M::STAGE_BYTES ? 0 : stage + M::STAGE_BYTES;
        }
        take(n_s - (steps - 1) * 4);
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 1));
            mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 2));
            if (tq == 0 && p < Tv) out[h][p] = __fmaf_rn(-sum[h], inv_cnt, mx[h]);
        }
    }
}

// The same for 32 positions, p the lane's, over every present key (score_mode 1): all lanes take the same row.
template <int D, int NH>
__device__ __forceinline__ void score_all(const __nv_bfloat16* const (&qh)[NH], const __nv_bfloat16* __restrict__ Kg,
                                          float* const (&out)[NH], const uint16_t* s_valid, uint32_t ring, int p, int p_end,
                                          int Tv) {
    using S = Sw<D>;
    using M = ScoreSmem<D>;
    const int lane = threadIdx.x & 31, row0 = lane / S::CPR, cc = lane % S::CPR;
    const float scale = rsqrtf((float)D), inv_cnt = 1.0f / (float)Tv;
    const int steps = (Tv + 31) / 32;
    auto fetch = [&](int step, uint32_t stage) {
        if (step < steps) {
#pragma unroll
            for (int i = 0; i < S::CPR; ++i) {
                const int r = i * (32 / S::CPR) + row0;
                ptx::cp_async_16(ring + stage + S::off(r, cc), Kg + (size_t)s_valid[min(step * 32 + r, Tv - 1)] * D + cc * 8);
            }
        }
        ptx::cp_async_commit();
    };
    __syncwarp();
#pragma unroll
    for (int s = 0; s < M::STAGES - 1; ++s) fetch(s, s * M::STAGE_BYTES);
    uint32_t q[NH][D / 2], stage = 0, ahead = M::RING_BYTES - M::STAGE_BYTES;
    load_queries<D, NH>(q, qh, s_valid[min(p, Tv - 1)]);
    float mx[NH], sum[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) { mx[h] = -INFINITY; sum[h] = 0.f; }
#pragma unroll 1
    for (int step = 0; step < steps; ++step) {
        ptx::cp_async_wait_group<M::STAGES - 2>();
        __syncwarp();
        fetch(step + M::STAGES - 1, ahead);
        const int n = min(32, Tv - step * 32);
#pragma unroll 2
        for (int j = 0; j < n; ++j) score_one_key<D, NH>(q, ring + stage, j, scale, mx, sum);
        ahead = stage;
        stage = stage == M::RING_BYTES - M::STAGE_BYTES ? 0 : stage + M::STAGE_BYTES;
    }
#pragma unroll
    for (int h = 0; h < NH; ++h)
        if (p < p_end) out[h][p] = __fmaf_rn(-sum[h], inv_cnt, mx[h]);
}

// grid B * Hk * n_blk * subs (blocks of a group together).  Dynamic smem: ScoreSmem.
//
// The scores decide which rows are active, so they are rounded as the one-launch form rounds them, whatever the data: fp32
// FMAs, four accumulators per dot product, the mean's sum in table order.  On the warp MMA the dot products take a tenth of
// the instructions, but they round in another order; ranking those and scoring the contested entries again is either not
// exact for keys with a large common part (a margin taken from the scores) or has contested entries in every other head (a
// margin proved from the rows' norms: the selection 15 -> 25 us) and thousands where scores tie.  Bound by the issue of 200
// instructions per 32 keys and two heads (0.57 per cycle and scheduler at 16 warps per SM) and by the shared-memory pipe
// (half busy): the tokens of a lane's copies come in one load (CPR loads: 2 to 7 % of the call more).  Whole calls on the MMA
// with a margin / here, us: 16 x 4096 tokens, d = 32: 82 / 80; 8 x 648, d = 64: 44 / 39; 1 x 4096, d = 32: 51 / 36; 64 x 2048:
// 170 / 175; 64 x 1024, d = 64: 130 / 140; 16 x 2048: 89 / 100; every key (score_mode 1), 32 x 1024, d = 32: 133 / 185.
template <int D, bool SAMPLED>
__global__ void __launch_bounds__(kSplitThreads, 2)
attend_split_score_kernel(const __grid_constant__ SplitArgs a, int subs) {
    extern __shared__ __align__(128) uint8_t s_raw[];
    __shared__ int red[kSplitWarps], s_hs[kMaxRK], s_khs[kMaxRK], s_rk;
    __shared__ int32_t s_kept[64];
    __shared__ float s_vs[kSplitWarps][D];
    using M = ScoreSmem<D>;
    uint16_t* s_valid = reinterpret_cast<uint16_t*>(s_raw + M::VALID_AT);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int grp = blockIdx.x / (a.n_blk * subs), sub = blockIdx.x % subs, blk = blockIdx.x / subs % a.n_blk;
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
            if (g == 0 && blk == 0 && sub == 0)
                for (int i = lane; i < a.k_h; i += 32) a.kept_out[(size_t)b * a.k_h + i] = s_kept[i];
            kept_row = s_kept;
        }
        bool bad;
        const int n = warp_group_heads(kept_row, a.k_h, a.Hq / a.Hk, g, a.Hq, s_hs, s_khs, bad);
        if (bad && blk == 0) atomicOr(a.status, SENTRY_STATUS_BIT_BAD_INDEX);
        if (lane == 0) s_rk = n;
    }
    const int Tv = list_present(a.ids, a.T, mask, s_valid, red, blk * kScoreBlock);
    __syncthreads();
    const int rk = s_rk;
    const int p_begin = blk * kScoreBlock, p_end = min(Tv, p_begin + kScoreBlock);
    if (g == 0 && sub == 0) {   // the list for the launches that follow
        for (int p = p_begin + threadIdx.x; p < p_end; p += kSplitThreads) a.valid[(size_t)b * a.T + p] = s_valid[p];
        if (blk == 0 && threadIdx.x == 0) a.tv[b] = Tv;
    }
    if (rk == 0) return;
    if (Tv == 0 && blk == 0 && threadIdx.x == 0) atomicOr(a.status, SENTRY_STATUS_BIT_EMPTY_MASK);
    if (p_begin >= Tv) return;
    if (sub == 0) {   // column sums of V over the positions: 16 bytes of a row per lane
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
    if (sub == 0 && threadIdx.x < D) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < kSplitWarps; ++w) t += s_vs[w][threadIdx.x];
        a.vsum[((size_t)grp * a.n_blk + blk) * D + threadIdx.x] = t;
    }
    if (a.given) return;

    // positions of this block to score
    const int p_share = kScoreBlock / subs, p_from = p_begin + sub * p_share, p_to = min(p_end, p_from + p_share);
    const int n_s = sentry_num_active(Tv, a.c);
    if (SAMPLED && (mask >= (uint32_t)a.n_subsets || a.offsets[mask] < 0)) {   // no table: every score ties
        if (threadIdx.x == 0) atomicOr(a.status, SENTRY_STATUS_BIT_BAD_INDEX);
        for (int h = 0; h < rk; ++h)
            for (int p = p_from + threadIdx.x; p < p_to; p += kSplitThreads)
                a.mscore[((size_t)b * a.k_h + s_khs[h]) * a.T + p] = 0.f;
        return;
    }
    uint16_t* s_tok = reinterpret_cast<uint16_t*>(s_raw + M::TOK_AT) + warp * kBatches * kBatchSteps * 32;
    const uint32_t ring = ptx::smem_u32(s_raw) + warp * M::RING_BYTES;
    const __nv_bfloat16* Kg = a.K + (size_t)grp * a.T * D;
    // sampled: a warp takes every eighth batch of the positions for all heads; all keys: 32 positions and a part of the heads
    int p0 = p_from + warp * kBatch, batches = (p_to - p0 + kBatch * kSplitWarps - 1) / (kBatch * kSplitWarps), h_begin = 0, h_end = rk;
    if constexpr (!SAMPLED) {
        const int chunks = p_share / 32, part = warp / chunks, per = (rk * chunks + kSplitWarps - 1) / kSplitWarps;
        p0 = p_from + warp % chunks * 32;
        h_begin = part * per;
        h_end = min(rk, h_begin + per);
    }
    if (p0 >= p_to) return;
    if constexpr (SAMPLED) stage_tokens<D / 8>(a.table + a.offsets[mask], a.score_mode, n_s, p0, batches, Tv, s_valid, s_tok, a.status);
    auto pass = [&](auto heads, int h0) {
        constexpr int NH = decltype(heads)::value;
        const __nv_bfloat16* qh[NH];
        float* out[NH];
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            qh[h] = a.Q + ((size_t)b * a.Hq + s_hs[h0 + h]) * a.T * D;
            out[h] = a.mscore + ((size_t)b * a.k_h + s_khs[h0 + h]) * a.T;
        }
        if constexpr (SAMPLED) score_sampled<D, NH>(qh, Kg, out, s_valid, s_tok, ring, n_s, p0 + (lane >> 2), batches, Tv);
        else score_all<D, NH>(qh, Kg, out, s_valid, ring, p0 + lane, p_to, Tv);
    };
    constexpr int HPP = D == 64 ? 2 : 4;            // heads per pass: their query rows live in registers
#pragma unroll 1
    for (int h0 = h_begin; h0 < h_end; h0 += HPP) {
        const int nh = min(HPP, h_end - h0);
        if (nh == 1) pass(std::integral_constant<int, 1>(), h0);
        else if (nh == 2) pass(std::integral_constant<int, 2>(), h0);
        else if constexpr (HPP == 4) {
            if (nh == 3) pass(std::integral_constant<int, 3>(), h0);
            else pass(std::integral_constant<int, 4>(), h0);
        }
    }
}

// ------------------------------------------------------------------------------------------ select
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
template <int KPT, int NW>
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
    bool cut = Tv == U;            // exactly U keys are >= t
    int bit = hi != lo ? (31 - __clz((int)(hi ^ lo))) | 1 : -1;   // digits of two bits, aligned
    uint32_t t = bit < 0 || cut ? lo : (bit == 31 ? 0u : hi & ~((2u << bit) - 1u));
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
    long long n = (3 * kSmCount + groups - 1) / groups;
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

int launch_select(sentry_ctx* ctx, const SplitArgs& p, cudaStream_t st) {
    const unsigned heads = (unsigned)p.B * p.k_h, packs = (heads + kSplitWarps - 1) / kSplitWarps;
    LaunchScope ls(ctx, KS_ATT_SELECT, st);
#define SELECT(KPT, NW, GRID) SENTRY_CUDA_TRY(launch_chained(attend_split_select_kernel<KPT, NW>, dim3(GRID), dim3(kSplitThreads), 0, st, p))
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
        // half the positions to a block while the blocks fit the GPU at once (two to an SM)
        const int subs = !p.given && (long long)groups * p.n_blk <= 2LL * ctx->sm_count ? 2 : 1;
        auto kern = d.score_mode != 1 ? attend_split_score_kernel<D, true> : attend_split_score_kernel<D, false>;
        const size_t smem = (size_t)ScoreSmem<D>::VALID_AT + list;
        if (smem > 46 * 1024)   // (beside the static arrays)
            SENTRY_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        LaunchScope ls(ctx, KS_ATT_SCORE, st);
        SENTRY_CUDA_TRY(launch_chained(kern, dim3(groups * (unsigned)(p.n_blk * subs)), dim3(kSplitThreads), smem, st, p, subs));
    }
    if (!p.given) {
        const int rc = launch_select(ctx, p, st);
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
