// Channel-compacted FFN (Section 4.6) for the d_model that the fused kernel of ffn_tc.cu does not take (its Y accumulator
// and an X tile must fit one SM beside the hidden tile: 128, 256, 384): any other multiple of 64 up to 1024, bf16 or fp16.
//
// Two tcgen05 GEMMs over the row plan, 128 x 128 tiles of one CTA each:
//   1  H = gelu(X[rows] . W1c^T)   X rows gathered by 16-byte async copies, W1c by TMA; exact erf
//   2  Y[rows] = H . W2c^T         both operands by TMA
// The hidden activations pass through a buffer of kWideTiles row tiles that stays in L2 (84 MB at 1280 channels); more
// rows than that go in turns.  They are stored as a 16-bit head plus a 16-bit remainder (h = hi + lo to 2^-17), and
// GEMM 2 multiplies both: what the plain-ALU kernel keeps in fp32 is not rounded to 16 bits here either.
//
// Tensor-bound in principle (6 D k_c operations per row with the remainder's product).  Measured on 3.7 k rows of
// d_model 768, 1229 channels in seven lists (33 row tiles): 32 + 25 us, 380 TFLOP/s of these operations, where the
// plain-ALU kernel (16 rows per CTA, one weight load per 16 multiply-adds) took 1065 us.
// Three 32 KB or two 48 KB stages let two CTAs share an SM, so that one's epilogue runs beside the other's arithmetic.
#include <cuda.h>
#include <math.h>

#include "common.cuh"
#include "ffn_plan.cuh"
#include "tc_common.cuh"
#include "ptx/sm100.cuh"

namespace {

constexpr int kWThreads = 256;
constexpr int kWBlock = 128 * 128;      // bytes of 128 rows x 64 elements
constexpr int kWideTiles = 128;         // row tiles the hidden buffer holds

template <bool FIRST>
struct WideCfg {
    static constexpr int BLOCKS = FIRST ? 2 : 3;            // operand blocks per stage: A, B or A head, A remainder, B
    static constexpr int STAGES = FIRST ? 3 : 2;
    static constexpr int STAGE_BYTES = BLOCKS * kWBlock;
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /* misc */ + 1024 /* alignment */;
};

struct WideMisc {
    uint64_t full[3], empty[3], acc_full;
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
__device__ __forceinline__ float gelu_exact(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752440f)); }

// grid (N tiles, row tiles of this turn).  FIRST: tm_b = W1c [lists * kc_pad, D], out_h / out_l = the hidden buffer's two
// planes.  Otherwise tm_a_hi / tm_a_lo = those planes, tm_b = W2c [lists * D, kc_pad], Y the result.
template <bool FIRST, bool F16>
__global__ void __launch_bounds__(kWThreads, 2)
ffn_wide_kernel(const __grid_constant__ CUtensorMap tm_a_hi, const __grid_constant__ CUtensorMap tm_a_lo,
                const __grid_constant__ CUtensorMap tm_b, const __nv_bfloat16* __restrict__ X, __nv_bfloat16* __restrict__ out_h,
                __nv_bfloat16* __restrict__ out_l, __nv_bfloat16* __restrict__ Y, FfnPlan plan, int n_lists, int tile0, int D,
                int kc_pad, unsigned int* status) {
    using C = WideCfg<FIRST>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = ptx::smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    WideMisc* misc = reinterpret_cast<WideMisc*>(smem_raw + (base - raw_addr) + C::STAGES * C::STAGE_BYTES);
    volatile int* abort_flag = &misc->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    grid_dependency_wait();
    int l, row0, n_rows;
    if (!ffn_tile_lookup(plan, n_lists, tile0 + (int)blockIdx.y, 128, l, row0, n_rows)) return;
    const int n0 = blockIdx.x * 128;                       // first output column
    const int KB = (FIRST ? D : kc_pad) / 64;              // 64-element K blocks

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
        ptx::tmem_alloc(ptx::smem_u32(&misc->tmem_base), 128);
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
                ptx::mbar_arrive_expect_tx(bar, FIRST ? kWBlock : 3 * kWBlock);
                if constexpr (!FIRST) {
                    ptx::tma_load_2d(dst, &tm_a_hi, kb * 64, (int)blockIdx.y * 128, bar);
                    ptx::tma_load_2d(dst + kWBlock, &tm_a_lo, kb * 64, (int)blockIdx.y * 128, bar);
                }
                ptx::tma_load_2d(dst + (C::BLOCKS - 1) * kWBlock, &tm_b, kb * 64, l * (FIRST ? kc_pad : D) + n0, bar);
            }
            __syncwarp();
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------------- UMMA issuer
        constexpr uint32_t idesc = F16 ? ptx::umma_idesc_f16(128, 128) : ptx::umma_idesc_bf16(128, 128);
        bool ok = true;
        for (int kb = 0; kb < KB && ok; ++kb) {
            const int s = kb % C::STAGES, use = kb / C::STAGES;
            ok = warp_wait(&misc->full[s], use & 1, abort_flag);
            if (!ok) break;
            ptx::tc_fence_after_sync();
            if (elect_one()) {
                const uint32_t a = base + s * C::STAGE_BYTES, b = a + (C::BLOCKS - 1) * kWBlock;
#pragma unroll
                for (int part = 0; part < C::BLOCKS - 1; ++part)
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        ptx::umma_bf16(tmem, ptx::umma_smem_desc_sw128(a + part * kWBlock + ks * 32),
                                       ptx::umma_smem_desc_sw128(b + ks * 32), idesc, (kb > 0 || part > 0 || ks > 0) ? 1u : 0u);
                ptx::umma_commit(ptx::smem_u32(&misc->empty[s]));
                if (kb == KB - 1) ptx::umma_commit(ptx::smem_u32(&misc->acc_full));
            }
            __syncwarp();
        }
    } else if (warp >= 4) {
        bool ok = true;
        if constexpr (FIRST) {
            // ------------------------------------------------------------ X row gather
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
        // -------------------------------------------------------------------- epilogue
        const int quarter = warp & 3, row = quarter * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
        const int n_cols = min(128, (FIRST ? kc_pad : D) - n0);
        int32_t yrow = -1;
        if (!FIRST && row < n_rows) yrow = (plan.rowout ? plan.rowout : plan.rowidx)[row0 + row];
        if (ok && warp_wait(&misc->acc_full, 0u, abort_flag)) {
            ptx::tc_fence_after_sync();
            const size_t hrow = ((size_t)blockIdx.y * 128 + row) * kc_pad + n0;
#pragma unroll 1
            for (int c0 = 0; c0 < n_cols; c0 += 32) {
                uint32_t r[32];
                ptx::tmem_ld_32x32(lane_base + c0, r);
                ptx::tmem_ld_wait();
                if constexpr (FIRST) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        uint32_t h[4], q[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float g0 = gelu_exact(__uint_as_float(r[8 * i + 2 * e])), g1 = gelu_exact(__uint_as_float(r[8 * i + 2 * e + 1]));
                            h[e] = pack_16x2<F16>(g0, g1);
                            q[e] = pack_16x2<F16>(g0 - lo_of<F16>(h[e]), g1 - hi_of<F16>(h[e]));
                        }
                        if (row < n_rows) {
                            *reinterpret_cast<uint4*>(out_h + hrow + c0 + 8 * i) = make_uint4(h[0], h[1], h[2], h[3]);
                            *reinterpret_cast<uint4*>(out_l + hrow + c0 + 8 * i) = make_uint4(q[0], q[1], q[2], q[3]);
                        }
                    }
                } else if (yrow >= 0) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        *reinterpret_cast<uint4*>(Y + (size_t)yrow * D + n0 + c0 + 8 * i) =
                            make_uint4(pack_16x2<F16>(__uint_as_float(r[8 * i]), __uint_as_float(r[8 * i + 1])),
                                       pack_16x2<F16>(__uint_as_float(r[8 * i + 2]), __uint_as_float(r[8 * i + 3])),
                                       pack_16x2<F16>(__uint_as_float(r[8 * i + 4]), __uint_as_float(r[8 * i + 5])),
                                       pack_16x2<F16>(__uint_as_float(r[8 * i + 6]), __uint_as_float(r[8 * i + 7])));
                }
            }
        }
    }
    tc_cta_teardown(abort_flag, status, tmem, 128);
}

template <bool F16>
int launch_wide(sentry_ctx* ctx, const FfnArgs& a, const FfnPlan& plan, void* w1c, void* w2c, int kc_pad, int max_tiles,
                void* hidden, cudaStream_t st) {
    const sentry_ffn_desc& d = a.d;
    const int turn = max_tiles < kWideTiles ? max_tiles : kWideTiles;
    __nv_bfloat16* hh = (__nv_bfloat16*)hidden;
    __nv_bfloat16* hl = hh + (size_t)turn * 128 * kc_pad;
    CUtensorMap m1, m2, ah, al;
    if (!make_weight_map(&m1, w1c, (uint64_t)d.n_lists * kc_pad, d.D, 128) ||
        !make_weight_map(&m2, w2c, (uint64_t)d.n_lists * d.D, kc_pad, 128) ||
        !make_weight_map(&ah, hh, (uint64_t)turn * 128, kc_pad, 128) || !make_weight_map(&al, hl, (uint64_t)turn * 128, kc_pad, 128))
        return SENTRY_ERR_CUDA;
    auto k1 = ffn_wide_kernel<true, F16>;
    auto k2 = ffn_wide_kernel<false, F16>;
    SENTRY_CUDA_TRY(cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, WideCfg<true>::SMEM_BYTES));
    SENTRY_CUDA_TRY(cudaFuncSetAttribute(k2, cudaFuncAttributeMaxDynamicSharedMemorySize, WideCfg<false>::SMEM_BYTES));
    for (int t0 = 0; t0 < max_tiles; t0 += turn) {
        const unsigned nt = (unsigned)(max_tiles - t0 < turn ? max_tiles - t0 : turn);
        LaunchScope ls(ctx, KS_FFN_MAIN, st, 2);
        SENTRY_CUDA_TRY(launch_chained(k1, dim3((unsigned)(kc_pad / 128), nt), dim3(kWThreads), (size_t)WideCfg<true>::SMEM_BYTES,
                                       st, ah, al, m1, (const __nv_bfloat16*)a.X, hh, hl, nullptr, plan, d.n_lists, t0, d.D,
                                       kc_pad, a.status));
        SENTRY_CUDA_TRY(launch_chained(k2, dim3((unsigned)((d.D + 127) / 128), nt), dim3(kWThreads),
                                       (size_t)WideCfg<false>::SMEM_BYTES, st, ah, al, m2, nullptr, nullptr, nullptr,
                                       (__nv_bfloat16*)a.Y, plan, d.n_lists, t0, d.D, kc_pad, a.status));
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
int launch_ffn_wide(sentry_ctx* ctx, const FfnArgs& a, const FfnPlan& plan, void* w1c, void* w2c, int kc_pad, int max_tiles,
                    void* hidden, cudaStream_t st) {
    return a.d.dtype == SENTRY_F16 ? launch_wide<true>(ctx, a, plan, w1c, w2c, kc_pad, max_tiles, hidden, st)
                                   : launch_wide<false>(ctx, a, plan, w1c, w2c, kc_pad, max_tiles, hidden, st);
}
