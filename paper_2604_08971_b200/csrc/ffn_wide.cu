// Channel-compacted FFN (Section 4.6) for the d_model that the fused kernel of ffn_tc.cu does not take (its Y accumulator
// and an X tile must fit one SM beside the hidden tile: 128, 256, 384): any other multiple of 64 up to 1024, bf16 or fp16.
//
// Two tcgen05 GEMMs over the row plan, a CTA per tile of 128 rows and BN columns:
//   1  H = gelu(X[rows] . W1c^T)   X rows gathered by 16-byte async copies, W1c by TMA
//   2  Y[rows] = H . W2c^T         both operands by TMA
// The hidden activations pass through a buffer of kWideTiles row tiles that stays in L2 (84 MB at 1280 channels); more
// rows than that go in turns.  They are stored as a 16-bit head plus a 16-bit remainder (h = hi + lo to 2^-17), and
// GEMM 2 multiplies both: what the plain-ALU kernel keeps in fp32 is not rounded to 16 bits here either.
//
// What bounds them: GEMM 1 its epilogue (two special-function and twenty other instructions per element, ffn_wide_math.cuh, by all
// eight warps; with the library's erff and four warps 6 us of 13 a tile) and its row gather, GEMM 2 the shared memory that serves the UMMAs'
// operands and the copies (128 bytes a cycle).  The column tile follows the number of row tiles, which only the device
// knows: small calls spread over more SMs, large ones read A less often.  GEMM 2 has one CTA per SM where an SM has a single
// tile, and two otherwise (wide_second_one has both sides): alone from the second tile on, with its epilogues beside
// nothing, it was slower than 128 x 128 tiles of two CTAs by up to 25 % (30 k rows of d_model 1024, 512 channels 549 -> 692 us; now 534).
// Measured, a call with its row plan on materialised weights, before (128 x 128 tiles, erff, four epilogue warps that stored row
// by row) and now: 3.7 k rows of d_model 768, 1229 channels in seven lists 56.7 -> 41.9 us; 524 rows, 765 channels 28.8 -> 22.8;
// 46 rows, 967 channels 27.1 -> 23.1; 233 rows of d_model 192, 340 channels 19.5 -> 15.3; 5.6 k rows, 384 channels 21.8 -> 18.4;
// 30.7 k rows of d_model 512, 1024 channels 185.0 -> 163.9.
// The GELU alone, as the erff form / the tail form without the polynomial / both parts (GEMM 2 with one CTA per SM throughout): 3.7 k
// rows 47.9 / 46.3 / 47.1; 30.7 k rows 191.4 / 182.7 / 187.5; 46 rows 24.9 / 24.6 / 24.8.
#include <cuda.h>
#include <math.h>

#include "common.cuh"
#include "ffn_plan.cuh"
#include "ffn_wide_math.cuh"
#include "tc_common.cuh"
#include "ptx/sm100.cuh"

namespace {

constexpr int kWThreads = 256;
constexpr int kWBlock = 128 * 128;      // bytes of 128 rows x 64 elements
constexpr int kWideTiles = 128;         // row tiles the hidden buffer holds

template <int FORM>
struct WideCfg {
    static constexpr bool FIRST = FORM == kWideFirst;
    static constexpr int A_BLOCKS = FIRST ? 1 : 2;          // A, or A's head and remainder
    static constexpr int BN_MAX = wide_bn_max(FORM);
    static constexpr int CTAS = wide_ctas(FORM);            // per SM
    static constexpr int STAGES = FIRST ? 3 : CTAS == 1 ? 4 : 2;
    static constexpr int STAGE_BYTES = A_BLOCKS * kWBlock + BN_MAX * 128;
    static constexpr int TMEM_COLS = 256;
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /* misc */ + 1024 /* alignment */;
};

struct WideMisc {
    uint64_t full[4], empty[4], acc_full;
    uint32_t tmem_base;
    int abort_flag;
};

template <bool F16>
__device__ __forceinline__ float lo_of(uint32_t w) {
    if constexpr (F16) return __half2float(__ushort_as_half((unsigned short)(w & 0xffffu)));
    else return __uint_as_float(w << 16);
}
template <bool F16>
__device__ __forceinline__ float hi_of(uint32_t w) {
    if constexpr (F16) return __half2float(__ushort_as_half((unsigned short)(w >> 16)));
    else return __uint_as_float(w & 0xffff0000u);
}
// Heads of a pair: the nearest values of the storage type, its largest one instead of inf.  A hidden value of up to twice that keeps a
// finite head and a remainder that makes up for it (an infinite head's remainder would be inf - inf).
template <bool F16>
__device__ __forceinline__ uint32_t pack_heads(float a, float b) {
    uint32_t v;
    if constexpr (F16) asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;" : "=r"(v) : "f"(b), "f"(a));
    else asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(v) : "f"(b), "f"(a));
    return v;
}
__device__ __forceinline__ float gelu_wide(float z) {
    return gelu_two_part(
        z,
        [](float x) {
            float y;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
            return y;
        },
        [](float x) {
            float y;
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
            return y;
        });
}

// grid: a CTA for every 64 columns of every row tile of this turn.  The tiles that there are at the width taken go to the first ones: with
// the idle ones among them a call of 59 row tiles, d_model 640, 500 channels took 38.2 us (now 33.1).
// FIRST: tm_b = W1c [lists * kc_pad, D], out_h / out_l = the hidden buffer's two planes.  Otherwise tm_a_hi / tm_a_lo = those
// planes, tm_b = W2c [lists * D, kc_pad], Y the result.
template <int FORM, bool F16>
__global__ void __launch_bounds__(kWThreads, WideCfg<FORM>::CTAS)
ffn_wide_kernel(const __grid_constant__ CUtensorMap tm_a_hi, const __grid_constant__ CUtensorMap tm_a_lo,
                const __grid_constant__ CUtensorMap tm_b, const __nv_bfloat16* __restrict__ X, __nv_bfloat16* __restrict__ out_h,
                __nv_bfloat16* __restrict__ out_l, __nv_bfloat16* __restrict__ Y, FfnPlan plan, int n_lists, int tile0, int turn,
                int D, int k_c, int kc_pad, int sm_count, unsigned int* status) {
    using C = WideCfg<FORM>;
    constexpr bool FIRST = C::FIRST;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = ptx::smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    WideMisc* misc = reinterpret_cast<WideMisc*>(smem_raw + (base - raw_addr) + C::STAGES * C::STAGE_BYTES);
    volatile int* abort_flag = &misc->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    grid_dependency_wait();
    const int kc = (k_c + 63) / 64 * 64;                   // channels that are computed (padded ones carry zero weights)
    const int cols = FIRST ? kc : D;
    const int row_tiles = min(plan.tile_start[n_lists] - tile0, turn);
    const int bn = wide_bn(FORM, row_tiles, cols, sm_count), across = (cols + bn - 1) / bn;
    const int tile = (int)blockIdx.x / across, n0 = ((int)blockIdx.x - tile * across) * bn;   // row tile, first output column
    int l, row0, n_rows;
    if (tile >= row_tiles || !ffn_tile_lookup(plan, n_lists, tile0 + tile, 128, l, row0, n_rows)) return;
    const int n_cols = min(bn, cols - n0);                 // a multiple of 32
    const int KB = (FIRST ? D : kc) / 64;                  // 64-element K blocks

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            ptx::mbar_init(ptx::smem_u32(&misc->full[s]), FIRST ? 5 : 1);   // the TMA's expect, and the four gathering warps
            ptx::mbar_init(ptx::smem_u32(&misc->empty[s]), 1);
        }
        ptx::mbar_init(ptx::smem_u32(&misc->acc_full), 1);
        misc->abort_flag = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 0) {
        ptx::tmem_alloc(ptx::smem_u32(&misc->tmem_base), C::TMEM_COLS);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem = misc->tmem_base;

    if (warp == 0) {
        // --------------------------------------------------------------- TMA producer
        bool ok = true;
        for (int kb = 0; kb < KB && ok; ++kb) {
            const int s = kb % C::STAGES, use = kb / C::STAGES;
            ok = warp_wait(&misc->empty[s], (use & 1) ^ 1, abort_flag);
            if (!ok) break;
            if (elect_one()) {
                const uint32_t bar = ptx::smem_u32(&misc->full[s]), dst = base + s * C::STAGE_BYTES;
                ptx::mbar_arrive_expect_tx(bar, (FIRST ? 0 : 2 * kWBlock) + n_cols * 128);
                if constexpr (!FIRST) {
                    ptx::tma_load_2d(dst, &tm_a_hi, kb * 64, tile * 128, bar);
                    ptx::tma_load_2d(dst + kWBlock, &tm_a_lo, kb * 64, tile * 128, bar);
                }
                for (int c = 0; c < n_cols; c += 32)
                    ptx::tma_load_2d(dst + C::A_BLOCKS * kWBlock + c * 128, &tm_b, kb * 64, l * (FIRST ? kc_pad : D) + n0 + c, bar);
            }
            __syncwarp();
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------------- UMMA issuer
        const uint32_t idesc = F16 ? ptx::umma_idesc_f16(128, n_cols) : ptx::umma_idesc_bf16(128, n_cols);
        bool ok = true;
        for (int kb = 0; kb < KB && ok; ++kb) {
            const int s = kb % C::STAGES, use = kb / C::STAGES;
            ok = warp_wait(&misc->full[s], use & 1, abort_flag);
            if (!ok) break;
            ptx::tc_fence_after_sync();
            if (elect_one()) {
                const uint32_t a = base + s * C::STAGE_BYTES, b = a + C::A_BLOCKS * kWBlock;
#pragma unroll
                for (int part = 0; part < C::A_BLOCKS; ++part)
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        ptx::umma_bf16(tmem, ptx::umma_smem_desc_sw128(a + part * kWBlock + ks * 32),
                                       ptx::umma_smem_desc_sw128(b + ks * 32), idesc, (kb > 0 || part > 0 || ks > 0) ? 1u : 0u);
                ptx::umma_commit(ptx::smem_u32(&misc->empty[s]));
                if (kb == KB - 1) ptx::umma_commit(ptx::smem_u32(&misc->acc_full));
            }
            __syncwarp();
        }
    } else if (FIRST && warp >= 4) {
        // ---------------------------------------------------------------- X row gather
        bool ok = true;
        const int tl = threadIdx.x - 128;
        int32_t rows[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int r = (tl + j * 128) >> 3;
            rows[j] = r < n_rows ? plan.rowidx[row0 + r] : -1;
        }
        int published = 0;
        auto publish = [&](int pending) {
            cp_async_wait_pending(pending);
            ptx::fence_proxy_async_smem();
            warp_arrive(&misc->full[published % C::STAGES]);
            ++published;
        };
        for (int kb = 0; kb < KB && ok; ++kb) {
            const int s = kb % C::STAGES, use = kb / C::STAGES;
            // a slot is refilled only when its block has been read, which needs every earlier block published
            if (kb >= C::STAGES)
                while (published <= kb - C::STAGES) publish(kb - published - 1);
            ok = warp_wait(&misc->empty[s], (use & 1) ^ 1, abort_flag);
            if (!ok) break;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int r = (tl + j * 128) >> 3, ci = tl & 7;
                const uint32_t dst = base + s * C::STAGE_BYTES + r * 128 + ((ci ^ (r & 7)) << 4);
                if (rows[j] >= 0) ptx::cp_async_16(dst, X + (size_t)rows[j] * D + kb * 64 + ci * 8);
                else asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(dst), "r"(0) : "memory");
            }
            ptx::cp_async_commit();
            if (kb - published >= 2) publish(2);
        }
        while (ok && published < KB) publish(KB - published - 1);
        ptx::cp_async_wait_all();
    }
    // -------------------------------------------------------------------- epilogue: all warps, two to a row, every other 32 columns
    // 32 columns at a time through 2 KB of the warp's own in the first stage (every UMMA has read it), so that a store writes
    // 64 consecutive bytes of eight rows.
    const int quarter = warp & 3, row = quarter * 32 + lane, half = warp >> 2;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    if (warp_wait(&misc->acc_full, 0u, abort_flag)) {
        ptx::tc_fence_after_sync();
        const uint32_t stg = base + (uint32_t)warp * 2048u;
        const uint32_t wr = stg + lane * 64, rd = stg + (lane >> 2) * 64;
        const uint32_t wx = (lane >> 1) & 3, rx = ((lane & 3) ^ ((lane >> 3) & 3)) << 4;
        int32_t grs[4];                                    // where the rows go that this lane stores pieces of
        {
            int32_t mine = -1;
            if (row < n_rows) mine = FIRST ? tile * 128 + row : (plan.rowout ? plan.rowout : plan.rowidx)[row0 + row];
#pragma unroll
            for (int i = 0; i < 4; ++i) grs[i] = __shfl_sync(0xffffffffu, mine, i * 8 + (lane >> 2));
        }
        auto store32 = [&](const uint32_t (&w)[16], __nv_bfloat16* dst, int ld) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(wr + ((i ^ wx) << 4)), "r"(w[4 * i]), "r"(w[4 * i + 1]),
                             "r"(w[4 * i + 2]), "r"(w[4 * i + 3])
                             : "memory");
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint4 v;
                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(rd + i * 512 + rx));
                if (grs[i] >= 0) *reinterpret_cast<uint4*>(dst + (size_t)grs[i] * ld + (lane & 3) * 8) = v;
            }
            __syncwarp();
        };
#pragma unroll 1
        for (int c0 = half * 32; c0 < n_cols; c0 += 64) {
            uint32_t r[32], w[16];
            ptx::tmem_ld_32x32(lane_base + c0, r);
            ptx::tmem_ld_wait();
            if constexpr (FIRST) {
                uint32_t q[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float g0 = gelu_wide(__uint_as_float(r[2 * i])), g1 = gelu_wide(__uint_as_float(r[2 * i + 1]));
                    w[i] = pack_heads<F16>(g0, g1);
                    q[i] = pack_16x2<F16>(g0 - lo_of<F16>(w[i]), g1 - hi_of<F16>(w[i]));
                }
                store32(w, out_h + n0 + c0, kc_pad);
                store32(q, out_l + n0 + c0, kc_pad);
            } else {
#pragma unroll
                for (int i = 0; i < 16; ++i) w[i] = pack_16x2<F16>(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
                store32(w, Y + n0 + c0, D);
            }
        }
    }
    tc_cta_teardown(abort_flag, status, tmem, C::TMEM_COLS);
}

template <bool F16>
int launch_wide(sentry_ctx* ctx, const FfnArgs& a, const FfnPlan& plan, void* w1c, void* w2c, int kc_pad, int max_tiles,
                void* hidden, cudaStream_t st) {
    const sentry_ffn_desc& d = a.d;
    const int turn = max_tiles < kWideTiles ? max_tiles : kWideTiles;
    __nv_bfloat16* hh = (__nv_bfloat16*)hidden;
    __nv_bfloat16* hl = hh + (size_t)turn * 128 * kc_pad;
    CUtensorMap m1, m2, ah, al;
    if (!make_weight_map(&m1, w1c, (uint64_t)d.n_lists * kc_pad, d.D, 32) ||
        !make_weight_map(&m2, w2c, (uint64_t)d.n_lists * d.D, kc_pad, 32) ||
        !make_weight_map(&ah, hh, (uint64_t)turn * 128, kc_pad, 128) || !make_weight_map(&al, hl, (uint64_t)turn * 128, kc_pad, 128))
        return SENTRY_ERR_CUDA;
    auto k1 = ffn_wide_kernel<kWideFirst, F16>;
    const bool one = wide_second_one(d.D, d.k_c, (max_tiles - d.n_lists) * 128LL, a.ids != nullptr, d.n_lists, kWideTiles, ctx->sm_count);
    auto k2 = one ? ffn_wide_kernel<kWideSecondOne, F16> : ffn_wide_kernel<kWideSecondTwo, F16>;
    constexpr size_t smem1 = WideCfg<kWideFirst>::SMEM_BYTES;
    const size_t smem2 = one ? WideCfg<kWideSecondOne>::SMEM_BYTES : WideCfg<kWideSecondTwo>::SMEM_BYTES;
    SENTRY_CUDA_TRY(cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem1));
    SENTRY_CUDA_TRY(cudaFuncSetAttribute(k2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2));
    for (int t0 = 0; t0 < max_tiles; t0 += turn) {
        const unsigned nt = (unsigned)(max_tiles - t0 < turn ? max_tiles - t0 : turn);
        LaunchScope ls(ctx, KS_FFN_MAIN, st, 2);
        SENTRY_CUDA_TRY(launch_chained(k1, dim3(nt * (unsigned)wide_grid_cols(d.k_c)), dim3(kWThreads), smem1, st, ah, al, m1,
                                       (const __nv_bfloat16*)a.X, hh, hl, nullptr, plan, d.n_lists, t0, (int)nt, d.D, d.k_c, kc_pad,
                                       ctx->sm_count, a.status));
        SENTRY_CUDA_TRY(launch_chained(k2, dim3(nt * (unsigned)wide_grid_cols(d.D)), dim3(kWThreads), smem2, st, ah, al, m2, nullptr,
                                       nullptr, nullptr, (__nv_bfloat16*)a.Y, plan, d.n_lists, t0, (int)nt, d.D, d.k_c, kc_pad,
                                       ctx->sm_count, a.status));
    }
    return SENTRY_OK;
}

}  // namespace

// The 16-bit types at the multiples of 64 that the fused kernel leaves.
bool ffn_wide_supported(const sentry_ffn_desc& d) {
    return (d.dtype == SENTRY_BF16 || d.dtype == SENTRY_F16) && d.D % 64 == 0 && d.D <= 1024 && !ffn_tc_supported(d);
}
int ffn_wide_kc_pad(int k_c) { return (k_c + 127) / 128 * 128; }
// The hidden buffer for a call of at most max_tiles row tiles.
size_t ffn_wide_hidden_bytes(int kc_pad, long long max_tiles) {
    return (size_t)(max_tiles < kWideTiles ? max_tiles : kWideTiles) * 128 * kc_pad * 2 * 2;
}
// CTAs of GEMM 1's first launch
long long ffn_wide_first_ctas(int k_c, long long max_tiles) {
    return (max_tiles < kWideTiles ? max_tiles : kWideTiles) * wide_grid_cols(k_c);
}
int launch_ffn_wide(sentry_ctx* ctx, const FfnArgs& a, const FfnPlan& plan, void* w1c, void* w2c, int kc_pad, int max_tiles,
                    void* hidden, cudaStream_t st) {
    return a.d.dtype == SENTRY_F16 ? launch_wide<true>(ctx, a, plan, w1c, w2c, kc_pad, max_tiles, hidden, st)
                                   : launch_wide<false>(ctx, a, plan, w1c, w2c, kc_pad, max_tiles, hidden, st);
}
