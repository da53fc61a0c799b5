// Pieces shared by the fused tcgen05 FFN kernels (ffn_tc.cu, ffn_tmem.cu): sizes, warp roles, UMMA issue and the zero rows.
#pragma once
#include "common.cuh"
#include "ffn_plan.cuh"
#include "tc_common.cuh"
#include "ptx/sm100.cuh"

namespace {

constexpr int kTileRows = 128;
constexpr int kBlockBytes = 128 * 128;   // 128 rows x 64 bf16: one X block, one hidden block
constexpr int kStageBytes = 2 * kBlockBytes;
constexpr int kStages = 3;
constexpr int kThreads = 512;
constexpr int kLoaderWarp0 = 3, kLoaderWarps = 4, kLoaderThreads = kLoaderWarps * 32;
constexpr int kEpiWarp0 = 7, kEpiWarps = 8;
constexpr int kZeroWarp = 15, kZeroBytes = 1024;   // zeros at the end of the misc block
constexpr int kTmemCols = 512;

// ---- lean forms for the single-thread roles -------------------------------------------------
// A warp that walks a chain of dependent scalar instructions with shared-memory round trips in
// it (an mbarrier probe, a flag poll, a vote) advances at 8 to 15 cycles per instruction here,
// so what the producers and issuers execute per stage is counted in instructions: barrier
// addresses are one add from a base, descriptors are a 32-bit add and a register pair, all the
// probes of a stage are issued back to back and voted on once.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);   // upper word of umma_smem_desc_sw128
__device__ __forceinline__ uint32_t desc_lo(uint32_t smem_addr) { return ((smem_addr >> 4) & 0x3fffu) | (1u << 16); }
// D (+)= A . B^T for one 128-byte K block = four 32-byte K steps (K = 16 16-bit or 32 8-bit elements);
// descriptors from their low words
#define SENTRY_MMA_KBLOCK(GROUP, KIND)                                                                                       \
    asm volatile(                                                                                                     \
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t.reg .b32 ta, tb;\n\t"                                            \
        "setp.ne.b32 p, %5, 0;\n\t"                                                                                   \
        "mov.b64 da, {%1, %4};\n\tmov.b64 db, {%2, %4};\n\t"                                                          \
        "tcgen05.mma.cta_group::" GROUP ".kind::" KIND " [%0], da, db, %3, p;\n\t"                                             \
        "setp.ne.b32 p, 1, 0;\n\t"                                                                                    \
        "add.u32 ta, %1, 2;\n\tadd.u32 tb, %2, 2;\n\tmov.b64 da, {ta, %4};\n\tmov.b64 db, {tb, %4};\n\t"              \
        "tcgen05.mma.cta_group::" GROUP ".kind::" KIND " [%0], da, db, %3, p;\n\t"                                             \
        "add.u32 ta, %1, 4;\n\tadd.u32 tb, %2, 4;\n\tmov.b64 da, {ta, %4};\n\tmov.b64 db, {tb, %4};\n\t"              \
        "tcgen05.mma.cta_group::" GROUP ".kind::" KIND " [%0], da, db, %3, p;\n\t"                                             \
        "add.u32 ta, %1, 6;\n\tadd.u32 tb, %2, 6;\n\tmov.b64 da, {ta, %4};\n\tmov.b64 db, {tb, %4};\n\t"              \
        "tcgen05.mma.cta_group::" GROUP ".kind::" KIND " [%0], da, db, %3, p;\n\t}"                                            \
        :                                                                                                             \
        : "r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(kDescHi), "r"(accumulate_first)                          \
        : "memory")
template <bool FP8>
__device__ __forceinline__ void mma_kblock(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc,
                                           uint32_t accumulate_first) {
    if constexpr (FP8) SENTRY_MMA_KBLOCK("1", "f8f6f4");
    else SENTRY_MMA_KBLOCK("1", "f16");
}
// Slow path of a stage's combined wait: the barriers one after the other, bounded (0 = none).
static __device__ __noinline__ bool wait_each_slow(uint32_t b0, uint32_t p0, uint32_t b1, uint32_t p1, uint32_t b2,
                                                   uint32_t p2, uint32_t b3, uint32_t p3, volatile int* abort_flag) {
    bool ok = ptx::mbar_wait(b0, p0, abort_flag);
    if (ok && b1 != 0u) ok = ptx::mbar_wait(b1, p1, abort_flag);
    if (ok && b2 != 0u) ok = ptx::mbar_wait(b2, p2, abort_flag);
    if (ok && b3 != 0u) ok = ptx::mbar_wait(b3, p3, abort_flag);
    return ok;
}

// Zero rows of Y for absent tokens, by one warp of every CTA; zsm = kZeroBytes of shared memory.
// The CTAs share the rows out evenly; runs of absent rows are written by bulk copies from a block of zeros, an
// instruction per kilobyte.  As blocks of the prepare launch these stores were a pass of their own over the absent
// part of Y (65 of 85 us at 4096 x 256 tokens, 3/7 absent); here they run beside the arithmetic.
template <int D>
__device__ __forceinline__ void ffn_zero_rows(const FfnPlan& plan, __nv_bfloat16* __restrict__ Y, uint32_t zsm) {
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < kZeroBytes / 16; i += 32)
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(zsm + i * 16), "r"(0) : "memory");
    ptx::fence_proxy_async_smem();
    __syncwarp();
    const int per = (plan.n_rows + (int)gridDim.x - 1) / (int)gridDim.x;
    const int r1 = min(plan.n_rows, ((int)blockIdx.x + 1) * per);
    for (int r0 = (int)blockIdx.x * per; r0 < r1; r0 += 128) {
        // 128 rows at a time: their ids and masks are requested together (a round trip per 32 rows made this warp
        // the last to finish)
        int m[4];
        uint32_t mask[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = min(r0 + u * 32 + lane, plan.n_rows - 1), bb = r / plan.Tlen;
            m[u] = __ldg(plan.zero_ids + (r - bb * plan.Tlen));
            mask[u] = __ldg(plan.zero_masks + bb);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool absent = r0 + u * 32 + lane < r1 && !(m[u] >= 0 && m[u] < 32 && ((mask[u] >> m[u]) & 1u));
            unsigned todo = __ballot_sync(0xffffffffu, absent);
            while (todo) {   // runs of absent rows: contiguous in Y, kZeroBytes per lane (32 rows are at most 24 KB)
                const int first = __ffs(todo) - 1;
                const unsigned rest = ~(todo >> first);
                const int len = rest ? min(__ffs(rest) - 1, 32 - first) : 32 - first;
                todo &= ~((len == 32 ? 0xffffffffu : (1u << len) - 1u) << first);
                const int off = lane * kZeroBytes, bytes = min(len * D * 2 - off, kZeroBytes);
                if (bytes > 0)
                    ptx::bulk_store(reinterpret_cast<uint8_t*>(Y) + (size_t)(r0 + u * 32 + first) * D * 2 + off, zsm,
                                    (uint32_t)bytes);
            }
        }
    }
    ptx::bulk_store_wait();   // the zeros have been read (and the rows are written before the grid ends)
}

}  // namespace
