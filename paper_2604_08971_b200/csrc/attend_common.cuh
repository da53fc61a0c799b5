// Device helpers shared by the bf16 SentryAttend kernels (Section 4.4): the swizzled row layout of
// K/V in shared memory, the sampled-score arithmetic and the top-U selections.
#pragma once
#include <math.h>

#include "common.cuh"
#include "ptx/sm100.cuh"

// The kernels that include this header exist twice: for bf16 tensors, and -- compiled again with
// SENTRY_ATT_F16 defined, under other entry-point names (attend_f16.cu, attend_long_f16.cu) -- for
// IEEE-half tensors.  The two builds differ only in the helpers below: the operand type of the
// mixed-precision FMA and of the warp MMA, and the 16-bit packing / unpacking.
#ifdef SENTRY_ATT_F16
#define ATT_PTX_TYPE "f16"
#define ATT_DTYPE SENTRY_F16
#else
#define ATT_PTX_TYPE "bf16"
#define ATT_DTYPE SENTRY_BF16
#endif

namespace {

// Low / high element of a packed 16-bit pair as fp32, and fp32 -> the 16 storage bits.
__device__ __forceinline__ float att_lo(uint32_t w) {
#ifdef SENTRY_ATT_F16
    return __half2float(__ushort_as_half((unsigned short)(w & 0xffffu)));
#else
    return __uint_as_float(w << 16);
#endif
}
__device__ __forceinline__ float att_hi(uint32_t w) {
#ifdef SENTRY_ATT_F16
    return __half2float(__ushort_as_half((unsigned short)(w >> 16)));
#else
    return __uint_as_float(w & 0xffff0000u);
#endif
}
__device__ __forceinline__ unsigned short att_bits(float x) {
#ifdef SENTRY_ATT_F16
    return __half_as_ushort(__float2half_rn(x));
#else
    return __bfloat16_as_ushort(__float2bfloat16_rn(x));
#endif
}

constexpr int kMaxRK = 4;          // kept heads of one KV group handled per CTA
constexpr int kScoreThreads = 256;
constexpr int kCoreThreads = 256;
constexpr int kCoreWarps = kCoreThreads / 32;
constexpr int kKeyTile = 64;
constexpr int kMaxActive = 48; // U <= 45 for T <= 8103 with c = 5 (checked on the host)
constexpr int kSmallT = 256;   // fused attention: sequences up to this length run in 128-thread CTAs
constexpr int kOrderMaxBatch = 1024; // batches up to this size are walked heaviest-sample-first

// Row layout in shared memory: rows of D bf16, 16-byte chunks XOR-swizzled so that both
// 8-consecutive-row matrix loads and random row gathers spread over the banks.
template <int D>
struct Sw {
    static constexpr int RB = D * 2;          // row bytes
    static constexpr int CPR = RB / 16;       // 16-byte chunks per row
    static constexpr int RPL = 128 / RB;      // rows per 128-byte line (>= 1 for D <= 64)
    __device__ static __forceinline__ uint32_t off(int row, int c) {
        return (uint32_t)row * RB + (uint32_t)((c ^ ((row / RPL) & (CPR - 1))) << 4);
    }
};

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}

// Kept heads of KV group g among kept_heads[b, :]: their head ids and kept-list slots.
__device__ __forceinline__ int group_heads(const int32_t* kept, int k_h, int r, int g, int Hq,
                                           int (&hs)[kMaxRK], int (&khs)[kMaxRK], bool& bad) {
    int rk = 0;
    bad = false;
    for (int j = 0; j < k_h; ++j) {
        const int h = kept[j];
        if (h < 0 || h >= Hq) { bad = true; continue; }
        if (h / r == g && rk < kMaxRK) { hs[rk] = h; khs[rk] = j; ++rk; }
    }
    return rk;
}

// The same by every warp for itself, a list entry to a lane (kept: shared or global memory; first: entry `lane`, 0 past the
// end).  The count is returned to all; the
// block's first warp leaves ids and slots in hs, khs (shared, complete behind the caller's next barrier): held in registers
// through the score pass they cost it 4 % at four CTAs per SM.
__device__ __forceinline__ int warp_heads(int first, const int32_t* kept, int k_h, int r, int g, int Hq, int* hs, int* khs,
                                          bool& bad) {
    const int lane = threadIdx.x & 31;
    int rk = 0;
    bad = false;
    for (int j0 = 0; j0 < k_h; j0 += 32) {
        const int h = j0 == 0 ? first : (j0 + lane < k_h ? kept[j0 + lane] : 0);
        const bool valid = h >= 0 && h < Hq, mine = j0 + lane < k_h && valid && h / r == g;
        bad |= __any_sync(0xffffffffu, !valid);
        const unsigned im = __ballot_sync(0xffffffffu, mine);
        const int at = rk + __popc(im & ((1u << lane) - 1u));
        if (threadIdx.x < 32 && mine && at < kMaxRK) { hs[at] = h; khs[at] = j0 + lane; }
        rk += __popc(im);
    }
    return min(rk, kMaxRK);
}

// The first four of a thread's tokens (positions u * blockDim + thread), requested before the sample's mask is known.
__device__ __forceinline__ void prefetch_ids(const int32_t* __restrict__ ids, int T, int (&id)[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int t = u * blockDim.x + threadIdx.x;
        id[u] = ids == nullptr ? 0 : (t < T ? __ldg(ids + t) : -1);
    }
}
// Present-token list of a sample, valid[p] = p-th present token, and kind[t] = present: four of a thread's tokens per round of
// counts (a round per blockDim tokens, with two barriers and a request each, took 6300 cycles of a CTA's 71000 at T = 1024,
// head selection included).  red: 64 ints; up to 16 warps.  Returns T_v.
__device__ __forceinline__ int block_list_present(const int32_t* __restrict__ ids, int T, uint32_t mask, int (&id)[4],
                                                  uint16_t* valid, uint8_t* kind, int* red) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int total = 0;
    for (int t0 = 0; t0 < T; t0 += 4 * blockDim.x) {
        if (t0 > 0) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int t = t0 + u * blockDim.x + threadIdx.x;
                id[u] = ids == nullptr ? 0 : (t < T ? __ldg(ids + t) : -1);
            }
            __syncthreads();                         // the counts of the round before have been read
        }
        const int rounds = min(4, (T - t0 + (int)blockDim.x - 1) / (int)blockDim.x);
        unsigned bm[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = t0 + u * blockDim.x + threadIdx.x;
            const bool ok = t < T && (ids == nullptr || (id[u] >= 0 && id[u] < 32 && ((mask >> id[u]) & 1u)));
            bm[u] = __ballot_sync(0xffffffffu, ok);
            if (t < T) kind[t] = ok;
            if (lane == 0 && u < rounds) red[u * nw + wid] = __popc(bm[u]);
        }
        __syncthreads();
        // counts in token order: entry u * nw + warp; a lane scans entries lane and lane + 32
        const int n = rounds * nw, c0 = lane < n ? red[lane] : 0, c1 = lane + 32 < n ? red[lane + 32] : 0;
        int s0 = c0, s1 = c1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, s0, o), b = __shfl_up_sync(0xffffffffu, s1, o);
            if (lane >= o) { s0 += a; s1 += b; }
        }
        const int half = __shfl_sync(0xffffffffu, s0, 31);
        const int e0 = total + s0 - c0, e1 = total + half + s1 - c1;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = u * nw + wid;
            const int base = e < 32 ? __shfl_sync(0xffffffffu, e0, e & 31) : __shfl_sync(0xffffffffu, e1, e & 31);
            if (u < rounds && ((bm[u] >> lane) & 1u))
                valid[base + __popc(bm[u] & ((1u << lane) - 1u))] = (uint16_t)(t0 + u * blockDim.x + threadIdx.x);
        }
        total += half + __shfl_sync(0xffffffffu, s1, 31);
    }
    __syncthreads();
    return total;
}

// ------------------------------------------------------------------------------------ score
// acc_lo += a.lo * b.lo, acc_hi += a.hi * b.hi for two bf16 pairs, in fp32: the mixed-precision
// FMA of sm_100 takes the bf16 operands as they are (exact products, fp32 accumulate), so
// neither the query nor the key row has to be unpacked to fp32 first.
__device__ __forceinline__ void fma_bf16_pair(float& acc_lo, float& acc_hi, uint32_t a, uint32_t b) {
    asm("{\n\t.reg .b16 al, ah, bl, bh;\n\t"
        "mov.b32 {al, ah}, %2;\n\tmov.b32 {bl, bh}, %3;\n\t"
        "fma.rn.f32." ATT_PTX_TYPE " %0, al, bl, %0;\n\tfma.rn.f32." ATT_PTX_TYPE " %1, ah, bh, %1;\n\t}"
        : "+f"(acc_lo), "+f"(acc_hi)
        : "r"(a), "r"(b));
}

// The first product of a sum: fma onto zero.
__device__ __forceinline__ void mul_bf16_pair(float& lo, float& hi, uint32_t a, uint32_t b) {
    asm("{\n\t.reg .b16 al, ah, bl, bh;\n\t"
        "mov.b32 {al, ah}, %2;\n\tmov.b32 {bl, bh}, %3;\n\t"
        "fma.rn.f32." ATT_PTX_TYPE " %0, al, bl, 0f00000000;\n\tfma.rn.f32." ATT_PTX_TYPE " %1, ah, bh, 0f00000000;\n\t}"
        : "=f"(lo), "=f"(hi)
        : "r"(a), "r"(b));
}

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32." ATT_PTX_TYPE "." ATT_PTX_TYPE ".f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// s = q . k / sqrt(d) for NH heads against one key row in shared memory; updates max and sum.
template <int D, int NH>
__device__ __forceinline__ void score_one_key(const uint32_t (&qw)[NH][D / 2], uint32_t row_addr_base, int row,
                                              float scale, float (&mx)[NH], float (&sum)[NH]) {
    using S = Sw<D>;
    float acc[NH][4];
#pragma unroll
    for (int h = 0; h < NH; ++h) acc[h][0] = acc[h][1] = acc[h][2] = acc[h][3] = 0.f;
#pragma unroll
    for (int cc = 0; cc < S::CPR; ++cc) {
        const uint4 v = lds128(row_addr_base + S::off(row, cc));
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            fma_bf16_pair(acc[h][0], acc[h][1], qw[h][4 * cc], v.x);
            fma_bf16_pair(acc[h][2], acc[h][3], qw[h][4 * cc + 1], v.y);
            fma_bf16_pair(acc[h][0], acc[h][1], qw[h][4 * cc + 2], v.z);
            fma_bf16_pair(acc[h][2], acc[h][3], qw[h][4 * cc + 3], v.w);
        }
    }
#pragma unroll
    for (int h = 0; h < NH; ++h) {
        const float sc = ((acc[h][0] + acc[h][1]) + (acc[h][2] + acc[h][3])) * scale;
        mx[h] = fmaxf(mx[h], sc);
        sum[h] += sc;
    }
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
#ifdef SENTRY_ATT_F16
    __half2 v = __floats2half2_rn(lo, hi);
#else
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
#endif
    return *reinterpret_cast<uint32_t*>(&v);
}
// bf16 pair of what the packed pair `head` = pack2(lo, hi) leaves of lo and hi
__device__ __forceinline__ uint32_t pack2_rem(float lo, float hi, uint32_t head) {
    return pack2(lo - att_lo(head), hi - att_hi(head));
}

// Warp-level top-k by radix selection over n order keys in shared memory (larger key first,
// ties -> lower index).  Writes remap[index] of the selected entries to out[0..k) in ascending
// index order.  `hist` = 256 ints of shared memory owned by this warp.
__device__ inline void warp_select_topk_radix(const uint32_t* keys, int n, int k, int32_t* out,
                                              const uint16_t* remap, int* hist) {
    const int lane = threadIdx.x & 31;
    uint32_t prefix = 0, fixed = 0;
    int want = k;
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int i = lane; i < 256; i += 32) hist[i] = 0;
        __syncwarp();
        for (int i = lane; i < n; i += 32) {
            const uint32_t key = keys[i];
            if ((key & fixed) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1);
        }
        __syncwarp();
        const int top = 255 - 8 * lane;      // this lane's digits, descending
        int mine = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) mine += hist[top - j];
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int above = incl - mine;
        const bool here = above < want && want <= incl;
        int digit = 0, rem = 0;
        if (here) {
            int acc = above;
            for (int j = 0; j < 8; ++j) {
                const int cdig = hist[top - j];
                if (want <= acc + cdig) { digit = top - j; rem = want - acc; break; }
                acc += cdig;
            }
        }
        const unsigned who = __ballot_sync(0xffffffffu, here);
        const int src = __ffs(who) - 1;
        digit = __shfl_sync(0xffffffffu, digit, src);
        rem = __shfl_sync(0xffffffffu, rem, src);
        prefix |= (uint32_t)digit << shift;
        fixed |= 255u << shift;
        want = rem;
        __syncwarp();
    }
    const uint32_t t = prefix;
    const int need_eq = want;
    int base = 0, eq_seen = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        const uint32_t key = i < n ? keys[i] : 0u;
        const bool is_eq = i < n && key == t, is_gt = i < n && key > t;
        const unsigned em = __ballot_sync(0xffffffffu, is_eq);
        const bool keep = is_gt || (is_eq && eq_seen + __popc(em & ((1u << lane) - 1u)) < need_eq);
        const unsigned km = __ballot_sync(0xffffffffu, keep);
        if (keep) out[base + __popc(km & ((1u << lane) - 1u))] = (int32_t)remap[i];
        base += __popc(km);
        eq_seen += __popc(em);
    }
    __syncwarp();
}

// Top-k of n <= 32 * KPL (up to 1023) order keys by ONE warp with the keys in registers (lane l holds keys l, l + 32, ...).
// The threshold is found two bits per step -- three candidates counted in one warp-wide add -- from the first bit in which
// the keys differ until exactly k keys lie from one on: 6 to 8 dependent adds, where one bit per step from the top took 32
// (attention of 256 samples of T <= 192: 28.7 -> 27.8 us).  Then the entries above it and, where keys tie at it, the first
// ties are compacted in ascending index order.  No shared-memory histograms, no atomics and no block barriers.
template <int KPL>
__device__ __forceinline__ void warp_select_topk_bits(const uint32_t* keys, int n, int k, int32_t* out,
                                                      const uint16_t* remap) {
    const int lane = threadIdx.x & 31;
    uint32_t r[KPL], hi = 0u, lo = 0xffffffffu;
#pragma unroll
    for (int j = 0; j < KPL; ++j) {
        const int i = j * 32 + lane;
        r[j] = i < n ? keys[i] : 0u;     // padding: below every candidate (candidates are >= 1)
        hi = max(hi, r[j]);
        if (i < n) lo = min(lo, r[j]);
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_min_sync(0xffffffffu, lo);
    bool cut = n == k;                                            // exactly k keys are >= t
    int bit = hi != lo ? (31 - __clz((int)(hi ^ lo))) | 1 : -1;   // digits of two bits, aligned
    uint32_t t = bit < 0 || cut ? lo : (bit == 31 ? 0u : hi & ~((2u << bit) - 1u));
#pragma unroll 1
    for (bit -= 1; bit >= 0 && !cut; bit -= 2) {
        const uint32_t c1 = t + (1u << bit), c2 = t + (2u << bit), c3 = t + (3u << bit);
        uint32_t cnt = 0u;                                        // from c1, c2, c3 on: ten bits each
#pragma unroll
        for (int j = 0; j < KPL; ++j) cnt += (r[j] >= c1 ? 1u : 0u) + (r[j] >= c2 ? 1u << 10 : 0u) + (r[j] >= c3 ? 1u << 20 : 0u);
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        const int k1 = (int)(cnt & 1023u), k2 = (int)(cnt >> 10) & 1023, k3 = (int)(cnt >> 20);
        if (k3 >= k) { t = c3; cut = k3 == k; }
        else if (k2 >= k) { t = c2; cut = k2 == k; }
        else if (k1 >= k) { t = c1; cut = k1 == k; }
    }
    int need_eq = n;                     // cut: every key equal to t is wanted
    if (!cut) {                          // t is the k-th largest key
        int gt = 0;
#pragma unroll
        for (int j = 0; j < KPL; ++j) gt += (r[j] > t) ? 1 : 0;
        need_eq = k - __reduce_add_sync(0xffffffffu, gt);
    }
    int base = 0, eq_seen = 0;
#pragma unroll
    for (int j = 0; j < KPL; ++j) {
        if (j * 32 >= n) break;          // warp-uniform
        const int i = j * 32 + lane;
        const bool is_eq = i < n && r[j] == t, is_gt = i < n && r[j] > t;
        const unsigned em = __ballot_sync(0xffffffffu, is_eq);
        const bool keep = is_gt || (is_eq && eq_seen + __popc(em & ((1u << lane) - 1u)) < need_eq);
        const unsigned km = __ballot_sync(0xffffffffu, keep);
        if (keep) out[base + __popc(km & ((1u << lane) - 1u))] = (int32_t)remap[i];
        base += __popc(km);
        eq_seen += __popc(em);
    }
    __syncwarp();
}
// Warp hh selects for head hh (keys [rk][stride], n <= 256 per head).
__device__ __forceinline__ void warps_select_topk_heads(const uint32_t* keys, int stride, int n, int k, int rk,
                                                        int32_t (*out)[kMaxActive], const uint16_t* remap) {
    const int warp = threadIdx.x >> 5;
    if (warp < rk) warp_select_topk_bits<8>(keys + (size_t)warp * stride, n, k, out[warp], remap);
}
// The same selection for the rk <= kMaxRK heads of a group at once, by the whole block: the threshold by counting digits of
// eight bits from the first bit in which a head's keys differ, until exactly k keys lie from it on (two counts as a rule; from
// the top bit, where most keys share a digit and the counters serialise, it took four, and a warp per head then went through
// all keys to put the selection in order: 10300 cycles of a CTA's 71000 at T = 1024, now 8000).  What lies from the threshold on is
// collected and put in order by rank; where keys tie at the threshold and not all of them are taken, a warp goes through the
// head's keys.  keys: [rk][stride] order keys, n per head; shared memory: hist kMaxRK * 256 ints, scratch kSelectScratch.
constexpr int kSelectScratch = 2 * kMaxRK * 32 + kMaxRK * kMaxActive + 5 * kMaxRK;
__device__ inline void block_select_topk_heads(const uint32_t* keys, int stride, int n, int k, int rk,
                                               int32_t (*out)[kMaxActive], const uint16_t* remap, int* hist, int* scratch) {
    uint32_t (*s_mm)[kMaxRK][32] = reinterpret_cast<uint32_t (*)[kMaxRK][32]>(scratch);   // [2] per warp: largest and smallest key
    int (*s_list)[kMaxActive] = reinterpret_cast<int (*)[kMaxActive]>(scratch + 2 * kMaxRK * 32);
    int* s_state = scratch + 2 * kMaxRK * 32 + kMaxRK * kMaxActive;
    uint32_t* s_prefix = reinterpret_cast<uint32_t*>(s_state);        // threshold: the bits that are known
    int *s_nb = s_state + kMaxRK, *s_want = s_nb + kMaxRK;            // bits that are not, keys still wanted among them
    int *s_done = s_want + kMaxRK, *s_n = s_done + kMaxRK;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = threadIdx.x; i < rk * 256; i += blockDim.x) hist[i] = 0;
    for (int hh = 0; hh < rk; ++hh) {
        uint32_t hi = 0u, lo = 0xffffffffu;
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const uint32_t key = keys[(size_t)hh * stride + i];
            hi = max(hi, key);
            lo = min(lo, key);
        }
        hi = __reduce_max_sync(0xffffffffu, hi);
        lo = __reduce_min_sync(0xffffffffu, lo);
        if (lane == 0) { s_mm[0][hh][warp] = hi; s_mm[1][hh][warp] = lo; }
    }
    __syncthreads();
    if (warp < rk) {
        const uint32_t hi = __reduce_max_sync(0xffffffffu, lane < nw ? s_mm[0][warp][lane] : 0u);
        const uint32_t lo = __reduce_min_sync(0xffffffffu, lane < nw ? s_mm[1][warp][lane] : 0xffffffffu);
        if (lane == 0) {
            const int nb = hi != lo ? 32 - __clz((int)(hi ^ lo)) : 0;
            s_prefix[warp] = n == k || nb == 32 ? 0u : hi >> nb << nb;
            s_nb[warp] = nb;
            s_want[warp] = k;
            s_n[warp] = 0;
            s_done[warp] = n == k ? 1 : (nb == 0 ? 2 : 0);   // 1: all keys from the threshold on, 2: ties at it are split
        }
    }
    __syncthreads();
    for (;;) {
        bool more = false;
        for (int hh = 0; hh < rk; ++hh) {
            if (s_done[hh]) continue;
            more = true;
            const uint32_t prefix = s_prefix[hh];
            const int nb = s_nb[hh], shift = max(nb - 8, 0);
            const uint32_t known = nb == 32 ? 0u : ~0u << nb, digit = (1u << (nb - shift)) - 1u;
            for (int i = threadIdx.x; i < n; i += blockDim.x) {
                const uint32_t key = keys[(size_t)hh * stride + i];
                if ((key & known) == prefix) atomicAdd(&hist[hh * 256 + ((key >> shift) & digit)], 1);
            }
        }
        if (!more) break;
        __syncthreads();
        if (warp < rk && !s_done[warp]) {
            int* h = hist + warp * 256;
            const int want = s_want[warp], shift = max(s_nb[warp] - 8, 0);
            const int top = 255 - 8 * lane;      // this lane's digits, descending
            int c[8], mine = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) { c[j] = h[top - j]; mine += c[j]; }
            int incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            int acc = incl - mine;
            if (acc < want && want <= incl) {    // exactly one lane
                int at = 0, cnt = 0;
                bool found = false;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (!found && want <= acc + c[j]) { found = true; at = j; cnt = c[j]; }
                    if (!found) acc += c[j];
                }
                s_prefix[warp] |= (uint32_t)(top - at) << shift;
                s_nb[warp] = shift;
                s_want[warp] = want - acc;
                s_done[warp] = cnt == want - acc ? 1 : (shift == 0 ? 2 : 0);
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) h[top - j] = 0;
        }
        __syncthreads();
    }
    for (int hh = 0; hh < rk; ++hh) {
        if (s_done[hh] != 1) continue;
        const uint32_t t = s_prefix[hh];
        for (int i = threadIdx.x; i < n; i += blockDim.x)
            if (keys[(size_t)hh * stride + i] >= t) s_list[hh][atomicAdd(&s_n[hh], 1)] = i;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < rk * 64; e += blockDim.x) {
        const int hh = e >> 6, a = e & 63;
        if (a >= k || s_done[hh] != 1) continue;
        const int mine = s_list[hh][a];
        int pos = 0;
        for (int b = 0; b < k; ++b) pos += s_list[hh][b] < mine ? 1 : 0;
        out[hh][pos] = (int32_t)remap[mine];
    }
    if (warp < rk && s_done[warp] == 2) {
        const uint32_t* kh = keys + (size_t)warp * stride;
        const uint32_t t = s_prefix[warp];
        const int need_eq = s_want[warp];
        int base = 0, eq_seen = 0;
        for (int i0 = 0; i0 < n; i0 += 32) {
            const int i = i0 + lane;
            const uint32_t key = i < n ? kh[i] : 0u;
            const bool is_eq = i < n && key == t, is_gt = i < n && key > t;
            const unsigned em = __ballot_sync(0xffffffffu, is_eq);
            const bool keep = is_gt || (is_eq && eq_seen + __popc(em & ((1u << lane) - 1u)) < need_eq);
            const unsigned km = __ballot_sync(0xffffffffu, keep);
            if (keep) out[warp][base + __popc(km & ((1u << lane) - 1u))] = (int32_t)remap[i];
            base += __popc(km);
            eq_seen += __popc(em);
        }
    }
}

}  // namespace
