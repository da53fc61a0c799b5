// Channel-compacted FFN on the 5th-generation tensor cores (Section 4.6), 16-bit operands at d_model 128 and 256: the
// hidden activations stay in tensor memory.
//
// One persistent CTA per SM walks tiles of 128 present rows (row table in ffn_plan.cuh).  Per tile and chunk of 128 kept
// channels (the last chunk of a list may be 64 wide):
//   GEMM1  H[128 x 128] = X_tile[128 x D] . W1c_chunk^T     (both operands in shared memory, fp32 in TMEM)
//   epilogue  H -> gelu -> 16 bits, written back over H in TMEM
//   GEMM2  Y[128 x D] += H . W2c_chunk                      (A operand read from TMEM)
// TMEM holds Y (D columns) and two hidden buffers of 128 columns, so GEMM1 of a chunk runs two chunks ahead of its GEMM2 and
// the tensor pipe does not wait for the epilogue.  All UMMAs come from one thread in the order G1(0) G1(1) G2(0) G1(2) G2(1)
// G1(3) ..., across tile boundaries too; G1(q + 2) reuses the buffer that G2(q), issued just before it, has read.
//
// What this buys: with the hidden tile in shared memory (ffn_tc.cu) there is room for one tile of X and one hidden buffer
// in TMEM, and at a tile boundary the next rows' fetch, the last GEMM2 and the stores of Y follow one another.  Without it two
// tiles of X fit (four at d_model 128), and what remains at a boundary is the drain of Y (about 1 us of a tile's 7).
//
// What bounds it: one CTA's shared memory (128 bytes a cycle) serves the UMMAs' operands and the TMA writes; at M = N = 128 a
// GEMM1 instruction reads as much as it can multiply, and a chunk of d_model 256 takes 2900 cycles for 2048 of arithmetic.  A
// pair of CTAs (P = 2, cta_group::2: 256 rows, each CTA holds half of every weight block) reads and fetches the weights once for
// both: 2300 cycles a chunk.  Per call with the row plan, hidden tile in shared memory / P = 1 / P = 2: 149 k rows, d_model 256,
// 512 channels 80 / 79 / 72 us; 599 k rows 303 / 298 / 270; 65 k rows 38.6 / 37.4 / 36.1; 37 k rows 26.2 / 24.4 / 25.5; 2.2 k rows
// 15.4 / 14.4 / 15.1; 35 k rows of d_model 128, 256 channels 16.7 / 14.1 / 16.0.  So pairs at d_model 256, where the weights are what is
// moved, from a number of rounds and chunks on (ffn_pair_rule.cuh), and single CTAs otherwise.
//
// Warp roles (512 threads): warp 0 = weight TMA producer (owns TMEM), warp 1 = UMMA issuer, warps 3-6 = X row gather, warps 7-14 =
// epilogue (two warps per TMEM lane quarter), warp 15 = zero rows of absent tokens.  Every wait is bounded; on expiry the CTA
// raises SENTRY_STATUS_BIT_TIMEOUT and unwinds.
#include <cuda.h>
#include <math.h>

#include "common.cuh"
#include "ffn_pair_rule.cuh"
#include "ffn_plan.cuh"
#include "ffn_tc_common.cuh"
#include "tc_common.cuh"
#include "ptx/sm100.cuh"

namespace {

// P: CTAs that share a tile's weights, each with 128 rows of its own: 1, or a pair (cta_group::2)
template <int D, int P>
struct TmCfg {
    static constexpr int CH = 128;                     // kept channels per chunk
    static constexpr int KB1 = D / 64;                 // X blocks per tile = K blocks of GEMM1
    static constexpr int NXS = 8;                      // X block slots
    static constexpr int NXB = NXS / KB1;              // tiles of X in flight
    static constexpr int NS = 3 * P;                   // weight stages
    static constexpr int STAGE_BYTES = kStageBytes / P;
    static constexpr int BLOCK_BYTES = kBlockBytes / P; // a K block of GEMM1's weights: 128 / P rows x 64 K
    static constexpr int H_COL0 = 256;                 // TMEM columns of the hidden buffers
    static constexpr int OFF_W = NXS * kBlockBytes;
    static constexpr int OFF_MISC = OFF_W + NS * STAGE_BYTES;
    static constexpr int SMEM_BYTES = OFF_MISC + 2048 + 1024;  // + misc + alignment slack
    static_assert(SMEM_BYTES <= 232448, "shared memory over the per-CTA limit");
};

struct TmMisc {
    uint64_t w_full[6], w_empty[6];
    uint64_t x_full[8];      // per block slot
    uint64_t x_empty[4];     // per tile of X
    uint64_t h_full[2];      // per hidden buffer
    uint64_t p_full[2];      // per hidden buffer: its 16-bit form is written
    uint64_t y_full, y_empty;
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(TmMisc) <= 2048 - kZeroBytes, "misc block too large");
#define TM_BAR(base, field) ((base) + (uint32_t)offsetof(TmMisc, field))

// D (+)= A . B^T over one 64-channel K block, A in tensor memory (8 columns per K = 16)
#define SENTRY_MMA_KBLOCK_TMEM(GROUP)                                                                       \
    asm volatile(                                                                                           \
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t.reg .b32 ta, tb;\n\t"                                      \
        "setp.ne.b32 p, %5, 0;\n\t"                                                                         \
        "mov.b64 db, {%2, %4};\n\t"                                                                         \
        "tcgen05.mma.cta_group::" GROUP ".kind::f16 [%0], [%1], db, %3, p;\n\t"                             \
        "setp.ne.b32 p, 1, 0;\n\t"                                                                          \
        "add.u32 ta, %1, 8;\n\tadd.u32 tb, %2, 2;\n\tmov.b64 db, {tb, %4};\n\t"                             \
        "tcgen05.mma.cta_group::" GROUP ".kind::f16 [%0], [ta], db, %3, p;\n\t"                             \
        "add.u32 ta, %1, 16;\n\tadd.u32 tb, %2, 4;\n\tmov.b64 db, {tb, %4};\n\t"                            \
        "tcgen05.mma.cta_group::" GROUP ".kind::f16 [%0], [ta], db, %3, p;\n\t"                             \
        "add.u32 ta, %1, 24;\n\tadd.u32 tb, %2, 6;\n\tmov.b64 db, {tb, %4};\n\t"                            \
        "tcgen05.mma.cta_group::" GROUP ".kind::f16 [%0], [ta], db, %3, p;\n\t}"                            \
        :                                                                                                   \
        : "r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(idesc), "r"(kDescHi), "r"(accumulate_first)              \
        : "memory")
template <int P>
__device__ __forceinline__ void mma_kblock_tmem_a(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t idesc,
                                                  uint32_t accumulate_first) {
    if constexpr (P == 2) SENTRY_MMA_KBLOCK_TMEM("2");
    else SENTRY_MMA_KBLOCK_TMEM("1");
}
template <int P>
__device__ __forceinline__ void mma_kblock_smem_a(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc,
                                                  uint32_t accumulate_first) {
    if constexpr (P == 2) SENTRY_MMA_KBLOCK("2", "f16");
    else SENTRY_MMA_KBLOCK("1", "f16");
}
template <int P>
__device__ __forceinline__ void commit(uint32_t bar) {
    if constexpr (P == 2) ptx::umma_commit_pair(bar);
    else ptx::umma_commit(bar);
}
// Walk over a CTA's tiles, ascending: P row tiles of a list make one tile, CTA `rank` has the rank-th of them (which may lie past
// the list's end: no rows).  The state moves on from list to list, so a step costs nothing while the list stays the same.
template <int P>
struct TileWalk {
    int l = -1, end = 0, first = 0;   // list, tiles up to its end, its first tile
    int r0 = 0, r1 = 0;               // its rows
    __device__ __forceinline__ void to(const FfnPlan& p, int tile) {
        while (tile >= end) {
            ++l;
            first = end;
            end += (p.tile_start[l + 1] - p.tile_start[l] + P - 1) / P;
            r0 = p.list_row0[l];
            r1 = p.list_row0[l + 1];
        }
    }
    __device__ __forceinline__ int row0(int tile, int rank) const { return r0 + ((tile - first) * P + rank) * kTileRows; }
    __device__ __forceinline__ int rows(int tile, int rank) const { return min(kTileRows, r1 - row0(tile, rank)); }
};

template <int D, bool F16, int P>
__global__ void __launch_bounds__(kThreads, 1)
ffn_tmem_kernel(const __grid_constant__ CUtensorMap tm_w1, const __grid_constant__ CUtensorMap tm_w1_64,
                const __grid_constant__ CUtensorMap tm_w2, const __nv_bfloat16* __restrict__ X, __nv_bfloat16* __restrict__ Y,
                FfnPlan plan, int n_lists, int k_c, int kc_pad, unsigned int* status) {
    using C = TmCfg<D, P>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = ptx::smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;   // 1024-byte aligned operand blocks
    TmMisc* misc = reinterpret_cast<TmMisc*>(smem_raw + (base - raw_addr) + C::OFF_MISC);
    const uint32_t xs = base, wsm = base + C::OFF_W;
    volatile int* abort_flag = &misc->abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = P == 2 ? (int)ptx::cluster_rank() : 0;    // CTA 0 of a pair issues the UMMAs of both
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::NS; ++s) {
            ptx::mbar_init(ptx::smem_u32(&misc->w_full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&misc->w_empty[s]), 1);
        }
        for (int s = 0; s < C::NXS; ++s) ptx::mbar_init(ptx::smem_u32(&misc->x_full[s]), P * kLoaderWarps);
        for (int s = 0; s < C::NXB; ++s) ptx::mbar_init(ptx::smem_u32(&misc->x_empty[s]), 1);
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(ptx::smem_u32(&misc->h_full[b]), 1);
            ptx::mbar_init(ptx::smem_u32(&misc->p_full[b]), P * kEpiWarps);
        }
        ptx::mbar_init(ptx::smem_u32(&misc->y_full), 1);
        ptx::mbar_init(ptx::smem_u32(&misc->y_empty), P * kEpiWarps);
        misc->abort_flag = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 0) {
        if constexpr (P == 2) {
            ptx::tmem_alloc_pair(ptx::smem_u32(&misc->tmem_base), kTmemCols);
            ptx::tmem_relinquish_pair();
        } else {
            ptx::tmem_alloc(ptx::smem_u32(&misc->tmem_base), kTmemCols);
            ptx::tmem_relinquish();
        }
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    if constexpr (P == 2) ptx::cluster_sync();   // the other CTA's barriers are initialised
    ptx::tc_fence_after_sync();
    const uint32_t tmem = misc->tmem_base;
    grid_dependency_wait();   // barriers and tensor memory are set up before the plan is there

    int n_tiles = plan.tile_start[n_lists];
    if constexpr (P == 2) {
        n_tiles = 0;
        for (int l = 0; l < n_lists; ++l) n_tiles += (plan.tile_start[l + 1] - plan.tile_start[l] + 1) / 2;
    }
    const int tile0 = (int)blockIdx.x / P, tile_step = (int)gridDim.x / P;
    const uint32_t mb = ptx::smem_u32(misc);
    const int NC = (k_c + C::CH - 1) / C::CH;
    const bool trim = (k_c - 1) % C::CH < 64;             // the last chunk has at most 64 channels: half of it is not computed
    const int my_tiles = (tile0 < n_tiles) ? (n_tiles - 1 - tile0) / tile_step + 1 : 0;
    // arrival of a warp at a barrier that the issuer waits for
    auto arrive_issuer = [&](uint32_t bar) {
        __syncwarp();
        if (lane == 0) {
            if constexpr (P == 2) ptx::mbar_arrive_cluster(ptx::cluster_addr(bar, 0));
            else ptx::mbar_arrive(bar);
        }
    };
    const uint32_t n_chunks = (uint32_t)(my_tiles * NC);
    // Ring order: step s = 0 .. n_chunks + 1 is GEMM2 of chunk s - 2, then GEMM1 of chunk s, as far as they exist.
    if (warp == 0) {
        // ------------------------------------------------------------ weight TMA producer
        if (elect_one()) {
            ptx::prefetch_tensormap(&tm_w1);
            ptx::prefetch_tensormap(&tm_w2);
            if (trim) ptx::prefetch_tensormap(&tm_w1_64);
        }
        __syncwarp();
        // one stage = one box, or two boxes a K block apart (x1 >= 0); in a pair each CTA fetches its half of the rows and
        // both halves count at CTA 0's barrier
        auto stage = [&](uint32_t n, const CUtensorMap* tm, int x0, int x1, int y, uint32_t bytes) -> bool {
            const uint32_t sl = n % C::NS, use = n / C::NS;
            const uint32_t we = TM_BAR(mb, w_empty) + 8u * sl;
            if (!__all_sync(0xffffffffu, ptx::mbar_try_wait(we, (use & 1u) ^ 1u)) &&
                !__all_sync(0xffffffffu, ptx::mbar_wait_slow(we, (use & 1u) ^ 1u, abort_flag)))
                return false;
            if (elect_one()) {
                const uint32_t bar = TM_BAR(mb, w_full) + 8u * sl;
                const uint32_t dst = wsm + sl * C::STAGE_BYTES;
                if (rank == 0) ptx::mbar_arrive_expect_tx(bar, bytes);
                if constexpr (P == 2) {
                    const uint32_t bar0 = ptx::cluster_addr(bar, 0);
                    ptx::tma_load_2d_pair(dst, tm, x0, y, bar0);
                    if (x1 >= 0) ptx::tma_load_2d_pair(dst + C::BLOCK_BYTES, tm, x1, y, bar0);
                } else {
                    ptx::tma_load_2d(dst, tm, x0, y, bar);
                    if (x1 >= 0) ptx::tma_load_2d(dst + C::BLOCK_BYTES, tm, x1, y, bar);
                }
            }
            __syncwarp();
            return true;
        };
        uint32_t n = 0;
        bool ok = true;
        int c1 = 0, c2 = 0;                      // chunk that GEMM1 / GEMM2 of this step work on
        int t1 = tile0, t2 = tile0;
        TileWalk<P> w1, w2;
#pragma unroll 1
        for (uint32_t s = 0; s < n_chunks + 2 && ok; ++s) {
            if (s >= 2) {
                if (c2 == 0) { w2.to(plan, t2); t2 += tile_step; }
                const int x = c2 * C::CH, y = w2.l * D + rank * (D / P);
                const bool half = trim && c2 == NC - 1;
                if constexpr (D == 256) {
                    ok = stage(n, &tm_w2, x, -1, y, kStageBytes);
                    ++n;
                    if (!half) {
                        if (ok) ok = stage(n, &tm_w2, x + 64, -1, y, kStageBytes);
                        ++n;
                    }
                } else {
                    ok = stage(n, &tm_w2, x, half ? -1 : x + 64, y, half ? kBlockBytes : kStageBytes);
                    ++n;
                }
                if (++c2 == NC) c2 = 0;
            }
            if (s < n_chunks && ok) {
                if (c1 == 0) { w1.to(plan, t1); t1 += tile_step; }
                const bool half = trim && c1 == NC - 1;
                const int y = w1.l * kc_pad + c1 * C::CH + rank * ((half ? 64 : C::CH) / P);
#pragma unroll
                for (int i = 0; i < C::KB1; i += 2, ++n)
                    if (ok)
                        ok = stage(n, half ? &tm_w1_64 : &tm_w1, 64 * i, 64 * i + 64, y, half ? kStageBytes / 2 : kStageBytes);
                if (++c1 == NC) c1 = 0;
            }
        }
        // the commits of CTA 0 arrive here too: none is outstanding when this CTA leaves
        if constexpr (P == 2)
            for (uint32_t k = n > (uint32_t)C::NS ? n - C::NS : 0u; k < n && ok; ++k)
                ok = warp_wait(&misc->w_empty[k % C::NS], (k / C::NS) & 1u, abort_flag);
    } else if (warp == 1 && rank == 0) {
        // ------------------------------------------------------------------- UMMA issuer
        // One thread issues every UMMA: the tensor pipe runs them in issue order, which is what lets GEMM1 of a chunk
        // overwrite the hidden buffer that the GEMM2 before it reads.
        constexpr uint32_t idesc128 = F16 ? ptx::umma_idesc_f16(128 * P, 128) : ptx::umma_idesc_bf16(128 * P, 128);
        constexpr uint32_t idesc64 = F16 ? ptx::umma_idesc_f16(128 * P, 64) : ptx::umma_idesc_bf16(128 * P, 64);
        constexpr uint32_t idescD = F16 ? ptx::umma_idesc_f16(128 * P, D) : ptx::umma_idesc_bf16(128 * P, D);
        constexpr uint32_t kXLo = kBlockBytes >> 4, kBlkLo = C::BLOCK_BYTES >> 4, kStageLo = C::STAGE_BYTES >> 4;
        const uint32_t xs_lo = desc_lo(xs), w_lo = desc_lo(wsm);
        bool ok = true;
        int c1 = 0, c2 = 0;
        uint32_t ti1 = 0, ti2 = 0;     // local tile of GEMM1 / GEMM2
        // the barriers of a stage: all probed back to back, then waited for one after the other
        auto wait_all = [&](uint32_t b0, uint32_t p0, uint32_t b1, uint32_t p1, uint32_t b2, uint32_t p2) -> bool {
            // (in a pair, the other CTA's copies and threads arrive on them too)
            auto probe = [&](uint32_t b, uint32_t ph_) { return P == 2 ? ptx::mbar_try_wait_cluster(b, ph_) : ptx::mbar_try_wait(b, ph_); };
            auto probe_all = [&]() {
                bool p = probe(b0, p0);
                if (b1 != 0u) p &= probe(b1, p1);
                if (b2 != 0u) p &= probe(b2, p2);
                return p;
            };
            if (!__all_sync(0xffffffffu, probe_all())) {
                if (!__all_sync(0xffffffffu, wait_each_slow(b0, p0, b1, p1, b2, p2, 0u, 0u, abort_flag))) return false;
                if constexpr (P == 2) probe_all();   // acquired at cluster scope too: no phase moves on before this warp does
            }
            ptx::tc_fence_after_sync();
            return true;
        };
        const uint32_t w_full = TM_BAR(mb, w_full), w_empty = TM_BAR(mb, w_empty);
        uint32_t sl = 0, ph = 0;          // ring slot and phase of the next stage
        auto step = [&]() {
            if (++sl == (uint32_t)C::NS) { sl = 0; ph ^= 1u; }
        };
#pragma unroll 1
        for (uint32_t s = 0; s < n_chunks + 2 && ok; ++s) {
            if (s >= 2) {
                // GEMM2 of chunk q = s - 2:  Y (+)= gelu(H) . W2c_chunk
                const uint32_t q = s - 2, buf = q & 1u;
                const bool first = c2 == 0, last = c2 == NC - 1, half = trim && last;
                const uint32_t pf = TM_BAR(mb, p_full) + 8u * buf, pp = (q >> 1) & 1u;
                const uint32_t ye = first ? TM_BAR(mb, y_empty) : 0u, yp = (ti2 & 1u) ^ 1u;
                const uint32_t hcol = tmem + C::H_COL0 + 128u * buf;
#pragma unroll
                for (int kb = 0; kb < (D == 256 ? 2 : 1); ++kb) {
                    if (!ok || (kb == 1 && half)) continue;
                    ok = kb == 0 ? wait_all(w_full + 8u * sl, ph, pf, pp, ye, yp) : wait_all(w_full + 8u * sl, ph, 0u, 0u, 0u, 0u);
                    if (!ok) continue;
                    if (elect_one()) {
                        const uint32_t b = w_lo + sl * kStageLo;
                        mma_kblock_tmem_a<P>(tmem, hcol + 64u * kb, b, idescD, (first && kb == 0) ? 0u : 1u);
                        if constexpr (D == 128)
                            if (!half) mma_kblock_tmem_a<P>(tmem, hcol + 64u, b + kBlkLo, idescD, 1u);
                        commit<P>(w_empty + 8u * sl);
                        if (last && (kb == (D == 256 ? 1 : 0) || half)) commit<P>(TM_BAR(mb, y_full));
                    }
                    __syncwarp();
                    step();
                }
                if (++c2 == NC) { c2 = 0; ++ti2; }
            }
            if (s < n_chunks && ok) {
                // GEMM1 of chunk s:  H = X . W1c_chunk^T
                const bool first = c1 == 0, half = trim && c1 == NC - 1;
                const uint32_t hcol = tmem + C::H_COL0 + 128u * (s & 1u);
                const uint32_t xb = (ti1 % C::NXB) * C::KB1, xp = (ti1 / C::NXB) & 1u;
                const uint32_t idesc = half ? idesc64 : idesc128;
#pragma unroll
                for (int i = 0; i < C::KB1; i += 2) {
                    if (!ok) continue;
                    const uint32_t xf = TM_BAR(mb, x_full) + 8u * (xb + i);
                    ok = wait_all(w_full + 8u * sl, ph, first ? xf : 0u, xp, first ? xf + 8u : 0u, xp);
                    if (!ok) continue;
                    if (elect_one()) {
                        const uint32_t a = xs_lo + (xb + i) * kXLo, b = w_lo + sl * kStageLo;
                        mma_kblock_smem_a<P>(hcol, a, b, idesc, i == 0 ? 0u : 1u);
                        mma_kblock_smem_a<P>(hcol, a + kXLo, b + kBlkLo, idesc, 1u);
                        commit<P>(w_empty + 8u * sl);
                        if (i == C::KB1 - 2) {
                            commit<P>(TM_BAR(mb, h_full) + 8u * (s & 1u));
                            if (c1 == NC - 1) commit<P>(TM_BAR(mb, x_empty) + 8u * (ti1 % C::NXB));
                        }
                    }
                    __syncwarp();
                    step();
                }
                if (++c1 == NC) { c1 = 0; ++ti1; }
            }
        }
    } else if (warp >= kLoaderWarp0 && warp < kEpiWarp0) {
        // ------------------------------------------------------------------ X row gather
        // Thread -> 8 (row, 16-byte piece) pairs of every 128 x 64 block, a row's 128 bytes by 8 lanes.  Up to three blocks
        // are in flight per thread; a block is published (x_full, one arrival per warp) once the copies of all lanes have
        // landed.
        constexpr int NJ = 1024 / kLoaderThreads;
        const int tl = threadIdx.x - kLoaderWarp0 * 32;
        TileWalk<P> walk;
        uint32_t gx = 0, published = 0;   // blocks issued / published by this warp
        bool ok = true;
        auto publish_oldest = [&]() {
            cp_async_wait_pending((int)(gx - published) - 1);
            ptx::fence_proxy_async_smem();
            if constexpr (P == 2) ptx::fence_release_smem_cluster();
            arrive_issuer(TM_BAR(mb, x_full) + 8u * (published % C::NXS));
            ++published;
        };
        for (int ti = 0; ti < my_tiles && ok; ++ti) {
            const int t = tile0 + ti * tile_step;
            walk.to(plan, t);
            const int row0 = walk.row0(t, rank), n_rows = walk.rows(t, rank);
            int32_t rows[NJ];
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const int r = (tl >> 3) + j * (kLoaderThreads / 8);
                rows[j] = r < n_rows ? plan.rowidx[row0 + r] : -1;
            }
            // never wait while holding blocks that the issuer may need
            uint64_t* bar = &misc->x_empty[ti % C::NXB];
            const uint32_t par = ((ti / C::NXB) & 1) ^ 1;
            while (gx > published && !__all_sync(0xffffffffu, ptx::mbar_test_wait(ptx::smem_u32(bar), par))) publish_oldest();
            ok = warp_wait(bar, par, abort_flag);
            if (!ok) break;
            const int ci = tl & 7;
            for (int kb = 0; kb < C::KB1; ++kb) {
                const uint32_t slot = gx % C::NXS;
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const int r = (tl >> 3) + j * (kLoaderThreads / 8);
                    const uint32_t dst = xs + slot * kBlockBytes + r * 128 + ((ci ^ (r & 7)) << 4);
                    if (rows[j] >= 0) ptx::cp_async_16(dst, X + (size_t)rows[j] * D + kb * 64 + ci * 8);
                    else asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(dst), "r"(0) : "memory");
                }
                ptx::cp_async_commit();
                ++gx;
                if (gx - published == 3) publish_oldest();
            }
            if (ti == 0)   // nothing is ahead of the first tile: its blocks do not wait for the next one's row table
                while (gx > published) publish_oldest();
        }
        while (ok && gx > published) publish_oldest();
        ptx::cp_async_wait_all();
    } else if (warp >= kEpiWarp0 && warp < kEpiWarp0 + kEpiWarps) {
        // ---------------------------------------------------------------------- epilogue
        const int ew = warp - kEpiWarp0;
        const int quarter = warp & 3, half = ew >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
        bool ok = true;
        uint32_t g = 0, ti = 0;
        // Y of a finished tile: TMEM -> 16 bits -> global.  A lane has a row; four lanes exchange their 16-byte pieces, so that
        // a store writes 64 consecutive bytes of eight rows (shared memory has no room for a staging block of Y: with one, and
        // four weight stages instead of six, the same time within 2 %; bulk copies of a row's pieces, 10 cycles each: 26 us more
        // on 149 k rows).
        auto drain_y = [&](uint32_t t_idx, int32_t grow) {
            if (!warp_wait(&misc->y_full, t_idx & 1u, abort_flag)) { ok = false; return; }
            ptx::tc_fence_after_sync();
            int32_t grs[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) grs[i] = __shfl_sync(0xffffffffu, grow, (lane & 28) + i);
#pragma unroll 1
            for (int pass = 0; pass < D / 128; ++pass) {
                uint32_t ra[32], rb[32];
                const uint32_t col0 = half * (D / 2) + pass * 64;
                ptx::tmem_ld_32x32(lane_base + col0, ra);
                ptx::tmem_ld_32x32(lane_base + col0 + 32u, rb);
                ptx::tmem_ld_wait();
                if (pass == D / 128 - 1) {
                    ptx::tc_fence_before_sync();
                    arrive_issuer(TM_BAR(mb, y_empty));
                }
#pragma unroll
                for (int g4 = 0; g4 < 2; ++g4) {
                    uint32_t u[4][4];      // pieces 4 g4 .. 4 g4 + 3 of this lane's row
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const uint32_t* r = g4 == 0 ? ra : rb;
                        u[i >> 2][i & 3] = pack_16x2<F16>(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
                    }
#pragma unroll
                    for (int b = 2; b > 0; b >>= 1)
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            if (j & b) continue;
                            const bool up = (lane & b) != 0;
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const uint32_t got = __shfl_xor_sync(0xffffffffu, up ? u[j][e] : u[j | b][e], b);
                                if (up) u[j][e] = got;
                                else u[j | b][e] = got;
                            }
                        }
                    // u[i] = this lane's piece (its number among the four) of row i of the four
                    __nv_bfloat16* dst = Y + col0 + g4 * 32 + (lane & 3) * 8;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (grs[i] >= 0) *reinterpret_cast<uint4*>(dst + (size_t)grs[i] * D) = make_uint4(u[i][0], u[i][1], u[i][2], u[i][3]);
                }
            }
        };
        TileWalk<P> walk;
        int32_t my_row = -1, prev_row = -1;
        for (; (int)ti < my_tiles && ok; ++ti) {
            const int t = tile0 + (int)ti * tile_step;
            walk.to(plan, t);
            prev_row = my_row;
            my_row = row < walk.rows(t, rank) ? (plan.rowout ? plan.rowout : plan.rowidx)[walk.row0(t, rank) + row] : -1;
            for (int c = 0; c < NC && ok; ++c, ++g) {
                const uint32_t buf = g & 1u;
                if (!warp_wait(&misc->h_full[buf], (g >> 1) & 1u, abort_flag)) { ok = false; break; }
                if (!(half == 1 && trim && c == NC - 1)) {
                    ptx::tc_fence_after_sync();
                    uint32_t h0[32], h1[32], pk[32];
                    const uint32_t tcol = lane_base + C::H_COL0 + 128u * buf + 64u * half;
                    ptx::tmem_ld_32x32(tcol, h0);
                    ptx::tmem_ld_32x32(tcol + 32, h1);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        pk[i] = gelu_pack_16x2<F16>(__uint_as_float(h0[2 * i]), __uint_as_float(h0[2 * i + 1]));
                        pk[16 + i] = gelu_pack_16x2<F16>(__uint_as_float(h1[2 * i]), __uint_as_float(h1[2 * i + 1]));
                    }
                    // in place, over the columns that only this warp reads
                    ptx::tmem_st_32x32(tcol, pk);
                    ptx::tmem_st_wait();
                    ptx::tc_fence_before_sync();
                }
                arrive_issuer(TM_BAR(mb, p_full) + 8u * buf);
                // Y of the previous tile is complete about now: its last GEMM2 was issued when the chunk before this one was ready
                if (c == 0 && ti > 0) drain_y(ti - 1, prev_row);
            }
        }
        if (ok && ti > 0) drain_y(ti - 1, my_row);
    } else if (warp == kZeroWarp && plan.zero_ids != nullptr) {
        ffn_zero_rows<D>(plan, Y, ptx::smem_u32(misc) + 2048u - kZeroBytes);
    }

    if constexpr (P == 2) ptx::cluster_sync();   // the pair's UMMAs read both CTAs' shared memory, its barriers hear from both
    tc_cta_teardown<P>(abort_flag, status, tmem, kTmemCols);
}

template <int D, bool F16, int P>
int launch_d(sentry_ctx* ctx, const FfnArgs& a, const FfnPlan& plan, void* w1c, void* w2c, int kc_pad, int max_tiles,
             cudaStream_t st) {
    using C = TmCfg<D, P>;
    const sentry_ffn_desc& d = a.d;
    CUtensorMap m1, m1h, m2;
    const uint64_t r1 = (uint64_t)d.n_lists * kc_pad, r2 = (uint64_t)d.n_lists * D;
    if (!make_weight_map(&m1, w1c, r1, D, 128 / P) || !make_weight_map(&m1h, w1c, r1, D, 64 / P) ||
        !make_weight_map(&m2, w2c, r2, kc_pad, D / P))
        return SENTRY_ERR_CUDA;
    auto kern = ffn_tmem_kernel<D, F16, P>;
    SENTRY_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES));
    int grid = P * (max_tiles < ctx->sm_count / P ? max_tiles : ctx->sm_count / P);
    if (grid < P) grid = P;
    LaunchScope ls(ctx, KS_FFN_MAIN, st);
    SENTRY_CUDA_TRY(launch_chained_clusters(P, kern, dim3(grid), dim3(kThreads), (size_t)C::SMEM_BYTES, st, m1, m1h, m2,
                                            (const __nv_bfloat16*)a.X, (__nv_bfloat16*)a.Y, plan, d.n_lists, d.k_c, kc_pad,
                                            a.status));
    return SENTRY_OK;
}

}  // namespace

bool ffn_tmem_supported(const sentry_ffn_desc& d) {
    return (d.dtype == SENTRY_BF16 || d.dtype == SENTRY_F16) && (d.D == 128 || d.D == 256);
}

int launch_ffn_tmem(sentry_ctx* ctx, const FfnArgs& a, const FfnPlan& plan, void* w1c, void* w2c, int kc_pad, int max_tiles,
                    cudaStream_t st) {
    const bool f16 = a.d.dtype == SENTRY_F16;
    if (a.d.D == 128) return f16 ? launch_d<128, true, 1>(ctx, a, plan, w1c, w2c, kc_pad, max_tiles, st)
                                 : launch_d<128, false, 1>(ctx, a, plan, w1c, w2c, kc_pad, max_tiles, st);
    if (ffn_takes_pairs(a.ids != nullptr, a.d.n_lists, a.d.k_c, max_tiles, ctx->sm_count))
        return f16 ? launch_d<256, true, 2>(ctx, a, plan, w1c, w2c, kc_pad, max_tiles, st)
                   : launch_d<256, false, 2>(ctx, a, plan, w1c, w2c, kc_pad, max_tiles, st);
    return f16 ? launch_d<256, true, 1>(ctx, a, plan, w1c, w2c, kc_pad, max_tiles, st)
               : launch_d<256, false, 1>(ctx, a, plan, w1c, w2c, kc_pad, max_tiles, st);
}
