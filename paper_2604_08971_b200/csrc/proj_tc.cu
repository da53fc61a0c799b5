// Projections of the pruned layer (Section 4.6, head pruning with GQA consistency) for bf16 on the 5th-generation tensor
// cores.  One CTA per (sample, tile of 128 present tokens, part of at most 256 output columns), two CTAs per SM: while one
// lists its tokens or stores its results, the other multiplies.
//
//   QKV   Every kept head, and K and V of every referenced KV group, is one "slice" of d columns.  A stage of the ring
//         holds 64 d_model indices of the tile's X rows (gathered, K-major) and of all the part's slices: their column
//         blocks W[64 rows, i d:(i+1) d] as they lie in memory (rows = d_model index, i.e. an MN-major B operand), so one
//         UMMA multiplies all of them and X is read from shared memory once per K step, not once per slice.  Pruned heads
//         and unreferenced groups are never fetched.
//   OUT   A stage holds one kept head: the tile's rows of its attention output (d wide) and the rows W_O[h d:(h+1) d] of
//         the part's columns.
// Before the stages warp 0 allocates tensor memory, warp 1 sets up barriers and slices and warps 2-7 list the tile's tokens, at
// once.  Then warp 0 feeds the weights by TMA, warp 1 issues the UMMAs, warps 4-7 gather the rows, and all eight store: 64
// accumulator columns at a time pass through shared memory so that eight lanes write 128 consecutive bytes.
// Bound by what a CTA does one after the other (19 K cycles at B = 128, T = 512, D = 384 with 15 slices of 32: 3.4 K to the
// first copy, 4.5 K until X and weights of the first stage are there, 7.5 K for six stages of 48 KB, two in flight, 3.5 K to
// store), which two CTAs per SM overlap in part.  One after the other with four storing warps, list and set-up took 2 and 3 K
// cycles: 128 x 512 tokens, 9 of 12 heads, QKV 63.4 -> 61.5 us, OUT 40.9 -> 37.7; 16 x 4096 at D = 256 46.5 -> 42.4 and 26.4 ->
// 20.9; 256 x 256 36.6 -> 35.4 and 22.9 -> 17.9.  Slower: two row tiles to a CTA that share the weights, one CTA per SM (63 ->
// 74 and 41 -> 53), three CTAs per SM with 128 columns (65 and 42; 46 -> 65 on 16 x 4096); without effect: box coordinates kept
// in registers (issue of a stage 1.2 -> 0.7 K cycles).
// A tile without a present token (missing modalities at T above 128) sets up and frees before it leaves, at once with its token
// count.  Calls full of them gained with the rest: 256 x 1024, 12 % present, QKV 29.0 -> 26.7 and OUT 47.4 -> 38.5; 16 x 4096,
// 3 % 15.0 -> 12.5 and 21.8 -> 14.3; 1024 x 256, 50 % 47.7 -> 48.0 and 54.2 -> 48.5.
// Measured there, the whole layer 262 -> 206 us: one CTA per SM that loaded X, multiplied slice by slice and then stored
// took 73 us for QKV and 61 for OUT.
// Every wait is bounded; on expiry the CTA raises SENTRY_STATUS_BIT_TIMEOUT and unwinds.
#include <cuda.h>

#include "attend_common.cuh"
#include "tc_common.cuh"

// Compiled a second time for IEEE-half tensors (proj_tc_f16.cu): the operand format of the UMMAs
// and the packing of the results (pack2, attend_common.cuh) are what differs.
#ifdef SENTRY_ATT_F16
#define PROJ_IDESC ptx::umma_idesc_f16_major
#else
#define PROJ_IDESC ptx::umma_idesc_bf16_major
#endif

namespace {

constexpr int kPThreads = 256, kPWarps = kPThreads / 32;
constexpr int kPCols = 256;                    // output columns of a part: two CTAs share the 512 columns of tensor memory
constexpr int kPRing = 96 * 1024;              // bytes of stages
constexpr int kPMaxStages = 8;
constexpr int kPSmem = kPRing + 1024;
constexpr int kMaxSlicesTc = 96;

struct ProjMisc {
    uint64_t full[kPMaxStages], empty[kPMaxStages], acc_full;
    uint32_t tmem_base;
    int abort_flag, n_slices, counts[kPWarps];
    int kind[kMaxSlicesTc], idx[kMaxSlicesTc];   // QKV: 0 = Q head, 1 = K group, 2 = V group.  OUT: kept-list slot, head
    uint16_t tok[128];                           // tokens of this tile
};

// The tile's tokens (present ones number 128 tt .. 128 tt + 127), by warps 2 to 7.  Every warp counts the present tokens of a run of
// 32-token pieces, eight of them requested at once; behind the CTA's barrier it writes the tokens of its run that are the
// tile's.  A run of at most eight pieces keeps its bits and is not read again.
constexpr int kListWarp0 = 2, kListWarps = kPWarps - kListWarp0;
struct TileList {
    int p0, p1, mine;
    unsigned bits[8];                            // of the pieces read last
    __device__ __forceinline__ void read(const int32_t* __restrict__ ids, int T, uint32_t mask, int pc) {
        const int lane = threadIdx.x & 31;
        int m[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int t = (pc + u) * 32 + lane;
            m[u] = pc + u < p1 && t < T ? __ldg(ids + t) : -1;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) bits[u] = __ballot_sync(0xffffffffu, m[u] >= 0 && m[u] < 32 && ((mask >> (m[u] & 31)) & 1u));
    }
    __device__ __forceinline__ void count(const int32_t* __restrict__ ids, int T, uint32_t mask, ProjMisc* misc) {
        const int w = (threadIdx.x >> 5) - kListWarp0, pieces = (T + 31) / 32, per = (pieces + kListWarps - 1) / kListWarps;
        p0 = min(w * per, pieces), p1 = min(p0 + per, pieces), mine = 0;
        for (int pc = p0; pc < p1; pc += 8) {
            read(ids, T, mask, pc);
#pragma unroll
            for (int u = 0; u < 8; ++u) mine += __popc(bits[u]);
        }
        if ((threadIdx.x & 31) == 0) misc->counts[w] = mine;
    }
    __device__ __forceinline__ void fill(const int32_t* __restrict__ ids, int T, uint32_t mask, int tt, ProjMisc* misc) {
        const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) - kListWarp0;
        int at = -tt * 128;
#pragma unroll
        for (int v = 0; v < kListWarps; ++v)
            if (v < w) at += misc->counts[v];
        if (at >= 128 || at + mine <= 0) return;
        for (int pc = p0; pc < p1; pc += 8) {
            if (p1 - p0 > 8) read(ids, T, mask, pc);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int r = at + __popc(bits[u] & ((1u << lane) - 1u));
                if (((bits[u] >> lane) & 1u) && r >= 0 && r < 128) misc->tok[r] = (uint16_t)((pc + u) * 32 + lane);
                at += __popc(bits[u]);
            }
        }
    }
};
// T_v of the sample, behind the barrier that follows TileList::count
__device__ __forceinline__ int present_tokens(const ProjMisc* misc) {
    int total = 0;
#pragma unroll
    for (int v = 0; v < kListWarps; ++v) total += misc->counts[v];
    return total;
}
// misc->tok is complete: among the warps that list (they gather next), and for warps 0 and 1, which read it with the results
__device__ __forceinline__ void list_done() {
    __syncwarp();
    asm volatile("bar.arrive 2, %0;" ::"n"(kPThreads) : "memory");
    asm volatile("bar.sync 1, %0;" ::"n"(kListWarps * 32) : "memory");
}
__device__ __forceinline__ void list_wait() {
    __syncwarp();
    asm volatile("bar.sync 2, %0;" ::"n"(kPThreads) : "memory");
}

// Barriers and the slice list of sample b (one warp; complete behind the caller's barrier).  Hk = 0: kept heads only.
__device__ __forceinline__ void proj_setup(ProjMisc* misc, int stages, const int32_t* __restrict__ kept, int k_h, int Hq, int Hk,
                                           unsigned int* status) {
    const int lane = threadIdx.x & 31;
    if (lane < stages) {
        ptx::mbar_init(ptx::smem_u32(&misc->full[lane]), 5);   // the TMA's expect, and the four gathering warps
        ptx::mbar_init(ptx::smem_u32(&misc->empty[lane]), 1);
    }
    if (lane == 0) {
        ptx::mbar_init(ptx::smem_u32(&misc->acc_full), 1);
        misc->abort_flag = 0;
    }
    ptx::fence_barrier_init();
    int n = 0;
    uint32_t groups = 0u;
    for (int j0 = 0; j0 < k_h; j0 += 32) {
        const int j = j0 + lane, h = j < k_h ? kept[j] : -1;
        const bool ok = h >= 0 && h < Hq;
        if (j < k_h && !ok) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
        const unsigned bm = __ballot_sync(0xffffffffu, ok);
        if (ok) {
            const int at = n + __popc(bm & ((1u << lane) - 1u));
            misc->kind[at] = Hk > 0 ? 0 : j;
            misc->idx[at] = h;
        }
        n += __popc(bm);
        groups |= __reduce_or_sync(0xffffffffu, ok && Hk > 0 ? 1u << (h / (Hq / Hk)) : 0u);
    }
    if ((groups >> lane) & 1u) {                 // (Hk is at most 32)
        const int at = n + 2 * __popc(groups & ((1u << lane) - 1u));
        misc->kind[at] = 1;
        misc->kind[at + 1] = 2;
        misc->idx[at] = misc->idx[at + 1] = lane;
    }
    n += 2 * __popc(groups);
    if (lane == 0) misc->n_slices = n;
}

// What a CTA does before its stages, at once: tensor memory (warp 0), barriers and slices (warp 1), the tokens counted (the rest).
// Returns T_v.
__device__ __forceinline__ int proj_prologue(ProjMisc* misc, TileList& list, const int32_t* __restrict__ kept, int k_h, int Hq, int Hk,
                                             const int32_t* __restrict__ ids, int T, uint32_t mask, unsigned int* status) {
    const int warp = threadIdx.x >> 5;
    if (warp == 0) {
        ptx::tmem_alloc(ptx::smem_u32(&misc->tmem_base), kPCols);
        ptx::tmem_relinquish();
    } else if (warp == 1) {
        proj_setup(misc, kPMaxStages, kept, k_h, Hq, Hk, status);
    } else {
        list.count(ids, T, mask, misc);
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    return present_tokens(misc);
}

// Gathers CPR 16-byte chunks of 128 rows per stage by warps 4-7: src(step, row, chunk) is the address or null (zeros),
// off(row, chunk) its place in the stage.  Returns false when a wait ran out.
template <int CPR, class Src, class Off>
__device__ __forceinline__ bool gather_steps(ProjMisc* misc, uint32_t ring, uint32_t stage_bytes, int stages, int steps, Src src,
                                             Off off, volatile int* abort_flag) {
    const int tl = threadIdx.x - 128, lag = min(stages - 1, 2);
    int published = 0, p_slot = 0;
    auto publish = [&](int pending) {
        cp_async_wait_pending(pending);
        ptx::fence_proxy_async_smem();
        warp_arrive(&misc->full[p_slot]);
        p_slot = p_slot + 1 == stages ? 0 : p_slot + 1;
        ++published;
    };
    bool ok = true;
    int slot = 0;
    uint32_t phase = 1u;
    for (int k = 0; k < steps; ++k) {
        // a slot is refilled only when its step has been read, which needs every earlier step published
        if (k >= stages)
            while (published <= k - stages) publish(k - published - 1);
        ok = warp_wait(&misc->empty[slot], phase, abort_flag);
        if (!ok) break;
#pragma unroll
        for (int j = 0; j < CPR; ++j) {
            const int i = tl + j * 128, r = i / CPR, cc = i % CPR;
            const uint32_t dst = ring + slot * stage_bytes + off(r, cc);
            const __nv_bfloat16* from = src(k, r, cc, j);
            if (from != nullptr) ptx::cp_async_16(dst, from);
            else asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(dst), "r"(0) : "memory");
        }
        ptx::cp_async_commit();
        if (k - published >= lag) publish(lag);
        if (++slot == stages) { slot = 0; phase ^= 1u; }
    }
    while (ok && published < steps) publish(steps - published - 1);
    ptx::cp_async_wait_all();
    return ok;
}

// 64 accumulator columns of the warp's 32 rows, rounded, to the warp's 4 KB of shared memory: 16-byte chunk c of row r at
// r * 128 + ((c ^ (r & 7)) << 4).
__device__ __forceinline__ void acc_to_smem(uint32_t taddr, uint32_t buf) {
    const int lane = threadIdx.x & 31;
    uint32_t acc[64];
    ptx::tmem_ld_32x32(taddr, reinterpret_cast<uint32_t(&)[32]>(acc[0]));
    ptx::tmem_ld_32x32(taddr + 32, reinterpret_cast<uint32_t(&)[32]>(acc[32]));
    ptx::tmem_ld_wait();
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) w[e] = pack2(__uint_as_float(acc[8 * c + 2 * e]), __uint_as_float(acc[8 * c + 2 * e + 1]));
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(buf + lane * 128 + ((c ^ (lane & 7)) << 4)), "r"(w[0]),
                     "r"(w[1]), "r"(w[2]), "r"(w[3])
                     : "memory");
    }
    __syncwarp();
}
__device__ __forceinline__ uint4 smem_chunk(uint32_t buf, int r, int c) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(buf + r * 128 + ((c ^ (r & 7)) << 4))
                 : "memory");
    return v;
}

// ------------------------------------------------------------------------------------- QKV
// grid B * tiles * parts (the parts of a tile together: the second one's X rows come from L2)
template <int DH>
__global__ void __launch_bounds__(kPThreads, 2)
proj_qkv_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                   const __grid_constant__ CUtensorMap tm_v, const __nv_bfloat16* __restrict__ X,
                   const int32_t* __restrict__ kept_heads, const int32_t* __restrict__ ids,
                   const uint32_t* __restrict__ masks, int Tlen, int D, int Hq, int Hk, int k_h, int tiles, int parts_max,
                   __nv_bfloat16* __restrict__ Q, __nv_bfloat16* __restrict__ K, __nv_bfloat16* __restrict__ V,
                   unsigned int* status) {
    constexpr int RB = DH * 2, NS = kPCols / DH;    // bytes of a slice row; slices of a part
    extern __shared__ uint8_t smem_raw[];
    __shared__ ProjMisc misc_s;
    ProjMisc* misc = &misc_s;
    const uint32_t ring = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    volatile int* abort_flag = &misc->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int part = blockIdx.x % parts_max, tile = blockIdx.x / parts_max, b = tile / tiles, tt = tile % tiles;
    const int KB = D / 64;
    if (warp == 0 && elect_one()) {
        ptx::prefetch_tensormap(&tm_q);
        ptx::prefetch_tensormap(&tm_k);
        ptx::prefetch_tensormap(&tm_v);
    }
    grid_dependency_wait();
    const uint32_t mask = masks[b];
    TileList list;
    const int Tv = proj_prologue(misc, list, kept_heads + (size_t)b * k_h, k_h, Hq, Hk, ids, Tlen, mask, status);
    const uint32_t tmem = misc->tmem_base;
    if (tt * 128 >= Tv) {                           // no present token in this tile
        tc_cta_teardown(abort_flag, status, tmem, kPCols);
        return;
    }
    const int n_rows = min(128, Tv - tt * 128);
    // equal shares of the slices for the parts that are needed
    const int n_all = misc->n_slices, parts = (n_all + NS - 1) / NS, per = parts > 0 ? (n_all + parts - 1) / parts : 0;
    const int s0 = part * per, n_sl = min(n_all - s0, per);
    if (n_sl > 0) {
        const uint32_t stage_bytes = 16384u + (uint32_t)n_sl * 64u * RB;
        const int stages = min(kPRing / (int)stage_bytes, kPMaxStages);
        bool ready = true;                          // this warp's part before the results went through
        if (warp == 0) {
            // -------------------------------------------------------- weights
            bool ok = true;
            int slot = 0;
            uint32_t phase = 1u;
            for (int kb = 0; kb < KB && ok; ++kb) {
                ok = warp_wait(&misc->empty[slot], phase, abort_flag);
                if (!ok) break;
                if (elect_one()) {
                    const uint32_t bar = ptx::smem_u32(&misc->full[slot]), dst = ring + slot * stage_bytes + 16384u;
                    ptx::mbar_arrive_expect_tx(bar, (uint32_t)n_sl * 64u * RB);
                    for (int j = 0; j < n_sl; ++j) {
                        const int kind = misc->kind[s0 + j];
                        ptx::tma_load_2d(dst + (uint32_t)j * 64u * RB, kind == 0 ? &tm_q : (kind == 1 ? &tm_k : &tm_v),
                                         misc->idx[s0 + j] * DH, kb * 64, bar);
                    }
                }
                __syncwarp();
                if (++slot == stages) { slot = 0; phase ^= 1u; }
            }
        } else if (warp == 1) {
            // ---------------------------------------------------------- UMMA issuer
            const uint32_t idesc = PROJ_IDESC(128, n_sl * DH, false, true);
            bool ok = true;
            int slot = 0;
            uint32_t phase = 0u;
            for (int kb = 0; kb < KB && ok; ++kb) {
                ok = warp_wait(&misc->full[slot], phase, abort_flag);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (elect_one()) {
                    const uint32_t a = ring + slot * stage_bytes, w = a + 16384u;
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        ptx::umma_bf16(tmem, ptx::umma_smem_desc_sw128(a + ks * 32),
                                       ptx::umma_smem_desc_rows(w + (uint32_t)ks * 16u * RB, RB, 64u * RB), idesc,
                                       (kb > 0 || ks > 0) ? 1u : 0u);
                    ptx::umma_commit(ptx::smem_u32(&misc->empty[slot]));
                    if (kb == KB - 1) ptx::umma_commit(ptx::smem_u32(&misc->acc_full));
                }
                __syncwarp();
                if (++slot == stages) { slot = 0; phase ^= 1u; }
            }
        } else {
            list.fill(ids, Tlen, mask, tt, misc);
            list_done();
        }
        if (warp < kListWarp0) list_wait();
        if (warp >= 4) {
            const __nv_bfloat16* rows[8];          // this thread's chunk of its rows
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int r = (threadIdx.x - 128 + j * 128) / 8;
                rows[j] = r < n_rows ? X + ((size_t)b * Tlen + misc->tok[r]) * D + (threadIdx.x & 7) * 8 : nullptr;
            }
            ready = gather_steps<8>(
                misc, ring, stage_bytes, stages, KB,
                [&](int kb, int, int, int j) { return rows[j] != nullptr ? rows[j] + kb * 64 : nullptr; },
                [](int r, int cc) { return (uint32_t)(r * 128 + ((cc ^ (r & 7)) << 4)); }, abort_flag);
        }
        // ----------------------------------------------------------------- results: two warps per 32 rows, blocks of 64 columns in turn
        if (ready && warp_wait(&misc->acc_full, 0u, abort_flag)) {
            ptx::tc_fence_after_sync();
            const int quarter = warp & 3, c = lane & 7;
            const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16), buf = ring + warp * 4096u;
            for (int c0 = (warp >> 2) * 64; c0 < n_sl * DH; c0 += 128) {
                acc_to_smem(taddr + c0, buf);
                const int s = (c0 + c * 8) / DH;                   // the slice of this lane's chunk
                if (s < n_sl) {
                    const int kind = misc->kind[s0 + s], idx = misc->idx[s0 + s];
                    __nv_bfloat16* dst = kind == 0 ? Q + ((size_t)b * Hq + idx) * Tlen * DH
                                                   : (kind == 1 ? K : V) + ((size_t)b * Hk + idx) * Tlen * DH;
                    dst += (c * 8) % DH;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int r = i * 4 + (lane >> 3);
                        if (quarter * 32 + r < n_rows)
                            *reinterpret_cast<uint4*>(dst + (size_t)misc->tok[quarter * 32 + r] * DH) = smem_chunk(buf, r, c);
                    }
                }
                __syncwarp();
            }
        }
    }
    tc_cta_teardown(abort_flag, status, tmem, kPCols);
}

// ------------------------------------------------------------------------------------- OUT
// grid B * tiles * parts; every CTA also clears its columns of the absent ones among token positions 128 tt ..
template <int DH>
__global__ void __launch_bounds__(kPThreads, 2)
proj_out_tc_kernel(const __grid_constant__ CUtensorMap tm_o, const __nv_bfloat16* __restrict__ A,
                   const int32_t* __restrict__ kept_heads, const int32_t* __restrict__ ids,
                   const uint32_t* __restrict__ masks, int Tlen, int D, int Hq, int k_h, int tiles, int parts,
                   __nv_bfloat16* __restrict__ out, unsigned int* status) {
    using S = Sw<DH>;
    constexpr uint32_t RB = DH * 2, kBox = DH * 128;   // bytes of an A row; of 64 columns of a head's rows of W_O
    extern __shared__ uint8_t smem_raw[];
    __shared__ ProjMisc misc_s;
    ProjMisc* misc = &misc_s;
    const uint32_t ring = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    volatile int* abort_flag = &misc->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int part = blockIdx.x % parts, tile = blockIdx.x / parts, b = tile / tiles, tt = tile % tiles;
    const int per = (D / 64 + parts - 1) / parts, box0 = part * per, n_box = min(D / 64 - box0, per);
    if (warp == 0 && elect_one()) ptx::prefetch_tensormap(&tm_o);
    grid_dependency_wait();
    const uint32_t mask = masks[b];
    // its columns of the absent ones among the 32 token positions from p on; m: the modality of position p + lane
    auto id_at = [&](int p) { return p + lane < Tlen ? __ldg(ids + p + lane) : -1; };
    auto clear_absent = [&](int p, int m) {
        unsigned gone = __ballot_sync(0xffffffffu, p + lane < Tlen && !(m >= 0 && m < 32 && ((mask >> m) & 1u)));
        const int pieces = n_box * 8, rows = pieces <= 16 ? 2 : 1;   // 16 bytes each; rows to a store
        const int second = rows == 2 && lane >= 16 ? 1 : 0, piece = lane - 16 * second;
        while (gone) {
            const int r0 = __ffs(gone) - 1;
            gone &= gone - 1;
            int r = r0;
            if (rows == 2 && gone) {
                if (second) r = __ffs(gone) - 1;
                gone &= gone - 1;
            }
            uint4* dst = reinterpret_cast<uint4*>(out + ((size_t)b * Tlen + p + r) * D) + box0 * 8;
            if (piece < pieces) dst[piece] = make_uint4(0, 0, 0, 0);
        }
    };
    // warps 2 and 3 clear beside the gathering ones; they ask for their positions' modalities with those of the token list
    // (behind it, and a row a store: 16 x 500 tokens at d_model 128, 5 of 8 heads of 16, a third of the tokens absent, 9.2 us, now 7.2)
    const int p_clear = tt * 128 + (warp - kListWarp0) * 32;
    int m_clear[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) m_clear[u] = warp == 2 || warp == 3 ? id_at(p_clear + u * 64) : -1;
    TileList list;
    const int Tv = proj_prologue(misc, list, kept_heads + (size_t)b * k_h, k_h, Hq, 0, ids, Tlen, mask, status);
    const uint32_t tmem = misc->tmem_base;
    if (tt * 128 >= Tv) {
        if (warp < 4) clear_absent(tt * 128 + warp * 32, id_at(tt * 128 + warp * 32));
        tc_cta_teardown(abort_flag, status, tmem, kPCols);
        return;
    }
    const int n_rows = min(128, Tv - tt * 128);
    const int n_sl = misc->n_slices;
    const uint32_t stage_bytes = 128u * RB + (uint32_t)n_box * kBox;
    const int stages = min(kPRing / (int)stage_bytes, kPMaxStages);
    bool ready = true;                              // this warp's part before the results went through
    if (warp == 0) {
        bool ok = true;
        int slot = 0;
        uint32_t phase = 1u;
        for (int s = 0; s < n_sl && ok; ++s) {
            ok = warp_wait(&misc->empty[slot], phase, abort_flag);
            if (!ok) break;
            if (elect_one()) {
                const uint32_t bar = ptx::smem_u32(&misc->full[slot]), dst = ring + slot * stage_bytes + 128u * RB;
                ptx::mbar_arrive_expect_tx(bar, (uint32_t)n_box * kBox);
                for (int i = 0; i < n_box; ++i)
                    ptx::tma_load_2d(dst + (uint32_t)i * kBox, &tm_o, (box0 + i) * 64, misc->idx[s] * DH, bar);
            }
            __syncwarp();
            if (++slot == stages) { slot = 0; phase ^= 1u; }
        }
    } else if (warp == 1) {
        const uint32_t idesc = PROJ_IDESC(128, n_box * 64, false, true);
        bool ok = true;
        int slot = 0;
        uint32_t phase = 0u;
        for (int s = 0; s < n_sl && ok; ++s) {
            ok = warp_wait(&misc->full[slot], phase, abort_flag);
            if (!ok) break;
            ptx::tc_fence_after_sync();
            if (elect_one()) {
                const uint32_t a = ring + slot * stage_bytes, w = a + 128u * RB;
#pragma unroll
                for (int ks = 0; ks < DH / 16; ++ks)
                    ptx::umma_bf16(tmem, ptx::umma_smem_desc_rows(a + ks * 32, RB),
                                   ptx::umma_smem_desc_rows(w + (uint32_t)ks * 16u * 128u, 128, kBox), idesc,
                                   (s > 0 || ks > 0) ? 1u : 0u);
                ptx::umma_commit(ptx::smem_u32(&misc->empty[slot]));
                if (s == n_sl - 1) ptx::umma_commit(ptx::smem_u32(&misc->acc_full));
            }
            __syncwarp();
            if (++slot == stages) { slot = 0; phase ^= 1u; }
        }
    } else {
        list.fill(ids, Tlen, mask, tt, misc);
        list_done();
        if (warp < 4) {
#pragma unroll
            for (int u = 0; u < 2; ++u) clear_absent(p_clear + u * 64, m_clear[u]);
        }
    }
    if (warp < kListWarp0) list_wait();
    if (warp >= 4) {
        const __nv_bfloat16* rows[S::CPR];
#pragma unroll
        for (int j = 0; j < S::CPR; ++j) {
            const int i = threadIdx.x - 128 + j * 128, r = i / S::CPR;
            rows[j] = r < n_rows ? A + ((size_t)b * k_h * Tlen + misc->tok[r]) * DH + (i % S::CPR) * 8 : nullptr;
        }
        ready = gather_steps<S::CPR>(
            misc, ring, stage_bytes, stages, n_sl,
            [&](int s, int, int, int j) {
                return rows[j] != nullptr ? rows[j] + (size_t)misc->kind[s] * Tlen * DH : nullptr;
            },
            [](int r, int cc) { return S::off(r, cc); }, abort_flag);
    }
    // results: two warps per 32 rows, boxes in turn
    if (ready && (n_sl == 0 || warp_wait(&misc->acc_full, 0u, abort_flag))) {
        ptx::tc_fence_after_sync();
        const int quarter = warp & 3, c = lane & 7;
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16), buf = ring + warp * 4096u;
        for (int i = warp >> 2; i < n_box; i += 2) {
            if (n_sl > 0) acc_to_smem(taddr + i * 64, buf);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int r = j * 4 + (lane >> 3);
                if (quarter * 32 + r < n_rows)   // (no valid kept head: the rows are zero)
                    *reinterpret_cast<uint4*>(out + ((size_t)b * Tlen + misc->tok[quarter * 32 + r]) * D + (box0 + i) * 64 + c * 8) =
                        n_sl > 0 ? smem_chunk(buf, r, c) : make_uint4(0, 0, 0, 0);
            }
            __syncwarp();
        }
    }
    tc_cta_teardown(abort_flag, status, tmem, kPCols);
}

template <int DH>
int launch_out_d(sentry_ctx* ctx, const ProjArgs& a, cudaStream_t st) {
    const sentry_proj_desc& d = a.d;
    CUtensorMap mo;
    if (!make_map_2d(&mo, a.WO, (uint64_t)d.Hq * DH, d.D, DH, 64)) return SENTRY_ERR_CUDA;
    auto kern = proj_out_tc_kernel<DH>;
    SENTRY_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kPSmem));
    const int tiles = (d.T + 127) / 128, parts = (d.D + kPCols - 1) / kPCols;
    LaunchScope ls(ctx, KS_PROJ_OUT, st);
    SENTRY_CUDA_TRY(launch_chained(kern, dim3((unsigned)((size_t)d.B * tiles * parts)), dim3(kPThreads), (size_t)kPSmem, st, mo,
                                   (const __nv_bfloat16*)a.A, a.kept_heads, a.ids, a.masks, d.T, d.D, d.Hq, d.k_h, tiles, parts,
                                   (__nv_bfloat16*)a.out, a.status));
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}

template <int DH>
int launch_qkv_d(sentry_ctx* ctx, const ProjArgs& a, cudaStream_t st) {
    const sentry_proj_desc& d = a.d;
    CUtensorMap mq, mk, mv;
    if (!make_map_2d(&mq, a.WQ, d.D, (uint64_t)d.Hq * DH, 64, DH) || !make_map_2d(&mk, a.WK, d.D, (uint64_t)d.Hk * DH, 64, DH) ||
        !make_map_2d(&mv, a.WV, d.D, (uint64_t)d.Hk * DH, 64, DH))
        return SENTRY_ERR_CUDA;
    auto kern = proj_qkv_tc_kernel<DH>;
    SENTRY_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kPSmem));
    const int tiles = (d.T + 127) / 128, groups = d.Hk < d.k_h ? d.Hk : d.k_h;   // at most: referenced groups
    const int parts = ((d.k_h + 2 * groups) * DH + kPCols - 1) / kPCols;
    LaunchScope ls(ctx, KS_PROJ_QKV, st);
    SENTRY_CUDA_TRY(launch_chained(kern, dim3((unsigned)((size_t)d.B * tiles * parts)), dim3(kPThreads), (size_t)kPSmem, st, mq, mk,
                                   mv, (const __nv_bfloat16*)a.X, a.kept_heads, a.ids, a.masks, d.T, d.D, d.Hq, d.Hk, d.k_h, tiles,
                                   parts, (__nv_bfloat16*)a.Q, (__nv_bfloat16*)a.K, (__nv_bfloat16*)a.V, a.status));
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}

}  // namespace

// bf16, head dim 16/32/64, d_model a multiple of 64.  The size clause describes no limit of this kernel: it is where an
// earlier one ended (96 KB of X and 72 KB of weights at d_model 384, d = 32), and it stays because Q and K decide which
// positions attention selects: beyond it the plain-ALU kernel's fp32 sums, in another order, are the result so far.  What
// that costs: 128 x 512 tokens at d_model 384 take 49 us here with 12 heads of 32, and 3690 us there with 6 heads of 64 (a
// CTA per token, which reads all kept weight columns).
bool project_qkv_tc_supported(const sentry_proj_desc& d) {
    if (d.dtype != ATT_DTYPE) return false;
    if (d.d != 16 && d.d != 32 && d.d != 64) return false;
    if (d.D % 64 != 0 || d.T > 65535) return false;
    if (d.k_h + 2 * d.Hk > kMaxSlicesTc) return false;
    const size_t list = ((size_t)d.T * 2 + 127) / 128 * 128;
    return (size_t)d.D * 256 + (size_t)3 * d.D * d.d * 2 + 1920 + list <= 220 * 1024;
}

int launch_project_qkv_tc(sentry_ctx* ctx, const ProjArgs& a, cudaStream_t st) {
    switch (a.d.d) {
        case 16: return launch_qkv_d<16>(ctx, a, st);
        case 32: return launch_qkv_d<32>(ctx, a, st);
        case 64: return launch_qkv_d<64>(ctx, a, st);
        default: return SENTRY_ERR_UNSUPPORTED;
    }
}

bool project_out_tc_supported(const sentry_proj_desc& d) {
    if (d.dtype != ATT_DTYPE) return false;
    if (d.d != 16 && d.d != 32 && d.d != 64) return false;
    return d.D % 64 == 0 && d.T <= 65535 && d.k_h <= kMaxSlicesTc;
}

int launch_project_out_tc(sentry_ctx* ctx, const ProjArgs& a, cudaStream_t st) {
    switch (a.d.d) {
        case 16: return launch_out_d<16>(ctx, a, st);
        case 32: return launch_out_d<32>(ctx, a, st);
        case 64: return launch_out_d<64>(ctx, a, st);
        default: return SENTRY_ERR_UNSUPPORTED;
    }
}
