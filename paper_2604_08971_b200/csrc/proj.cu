// Projections of the pruned layer (Section 4.6, "Head pruning with GQA consistency"): only the
// column blocks of W_Q that belong to the kept heads, only the blocks of W_K / W_V of the KV groups
// those heads reference, only the row blocks of W_O of the kept heads, and only present tokens.
//   Q[b,h,t,:] = x_t . W_Q[:, h d:(h+1) d]  (h kept)      K, V[b,g,t,:] likewise (g referenced)
//   out[b,t,:] = sum_j A[b,j,t,:] . W_O[h_j d:(h_j+1) d, :]
// This file: the plain-ALU form (any dtype, fp32 accumulation), one CTA per token.
#include "common.cuh"

namespace {

constexpr int kProjThreads = 256;
constexpr int kMaxSlices = 128;  // kept heads (at most 64) + 2 x referenced groups (at most 32)

// Bound by the weight columns' round trips, so by the CTAs that an SM holds: four, at 64 registers.  Left to itself the compiler takes 80
// and fewer loads on the way: 500 tokens of d_model 768, 7 of 12 heads of 64, 336 us (now 126, and 128 before the slice list was made by a
// warp), 64 k tokens 25.0 ms (12.8, 13.4); fp32, 1600 tokens of d_model 64, 13.9 us (11.8, 14.7).
template <typename T>
__global__ void __launch_bounds__(kProjThreads, 4)
project_qkv_kernel(const T* __restrict__ X, const T* __restrict__ WQ, const T* __restrict__ WK,
                   const T* __restrict__ WV, const int32_t* __restrict__ kept_heads,
                   const int32_t* __restrict__ ids, const uint32_t* __restrict__ masks, int Tlen, int D, int Hq,
                   int Hk, int d, int k_h, T* __restrict__ Q, T* __restrict__ K, T* __restrict__ V,
                   unsigned int* status) {
    extern __shared__ float s_x[];                 // [D]
    __shared__ int s_kind[kMaxSlices], s_idx[kMaxSlices], s_n;
    grid_dependents_start_if_small();
    grid_dependency_wait();
    const int b = blockIdx.x / Tlen, t = blockIdx.x % Tlen;
    // the list entry and the row are requested together with what tells whether the token is there
    const int lane = threadIdx.x & 31;
    const int h_mine = threadIdx.x < 32 && lane < k_h ? kept_heads[(size_t)b * k_h + lane] : 0;
    const T* x = X + ((size_t)b * Tlen + t) * D;
    const float x_mine = (int)threadIdx.x < D ? to_f32<T>(x[threadIdx.x]) : 0.f;
    const int m = ids[t];
    if (m < 0 || m >= 32 || !((masks[b] >> m) & 1u)) return;       // absent token: nothing is written
    if (threadIdx.x < 32) {
        // slices: one per kept head (Q), one K and one V per referenced group
        const int r = Hq / Hk;
        int n = 0;
        uint32_t groups = 0;
        for (int j0 = 0; j0 < k_h; j0 += 32) {
            const int j = j0 + lane, h = j0 == 0 ? h_mine : (j < k_h ? kept_heads[(size_t)b * k_h + j] : 0);
            const bool valid = h >= 0 && h < Hq, in = j < k_h && valid;
            if (j < k_h && !valid) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
            const unsigned im = __ballot_sync(0xffffffffu, in);
            if (in) { const int at = n + __popc(im & ((1u << lane) - 1u)); s_kind[at] = 0; s_idx[at] = h; }
            n += __popc(im);
            groups |= __reduce_or_sync(0xffffffffu, in ? 1u << (h / r) : 0u);
        }
        const bool in = lane < Hk && ((groups >> lane) & 1u);
        if (in) {
            const int at = n + 2 * __popc(groups & ((1u << lane) - 1u));
            s_kind[at] = 1; s_idx[at] = lane;
            s_kind[at + 1] = 2; s_idx[at + 1] = lane;
        }
        if (lane == 0) s_n = n + 2 * __popc(groups);
    }
    for (int e = threadIdx.x; e < D; e += blockDim.x) s_x[e] = e == (int)threadIdx.x ? x_mine : to_f32<T>(x[e]);
    __syncthreads();
    const int total = s_n * d;
    for (int o = threadIdx.x; o < total; o += blockDim.x) {
        const int sl = o / d, c = o % d;
        const int kind = s_kind[sl], idx = s_idx[sl];
        const T* W = kind == 0 ? WQ : (kind == 1 ? WK : WV);
        const int ld = (kind == 0 ? Hq : Hk) * d;
        const int col = idx * d + c;
        float acc = 0.f;
#pragma unroll 16
        for (int e = 0; e < D; ++e) acc = fmaf(s_x[e], to_f32<T>(W[(size_t)e * ld + col]), acc);
        T* dst = kind == 0 ? Q + (((size_t)b * Hq + idx) * Tlen + t) * d
                           : (kind == 1 ? K : V) + (((size_t)b * Hk + idx) * Tlen + t) * d;
        dst[c] = from_f32<T>(acc);
    }
}

template <typename T>
__global__ void __launch_bounds__(kProjThreads)
project_out_kernel(const T* __restrict__ A, const T* __restrict__ WO, const int32_t* __restrict__ kept_heads,
                   const int32_t* __restrict__ ids, const uint32_t* __restrict__ masks, int Tlen, int D, int Hq,
                   int d, int k_h, T* __restrict__ out, unsigned int* status) {
    extern __shared__ float s_a[];                 // [k_h * d]
    __shared__ int s_h[64];
    grid_dependents_start_if_small();
    grid_dependency_wait();
    const int b = blockIdx.x / Tlen, t = blockIdx.x % Tlen;
    T* o = out + ((size_t)b * Tlen + t) * D;
    const int n_a = k_h * d, i_mine = min((int)threadIdx.x, n_a - 1);   // (requested with the mask; of an absent token, not used)
    const float a_mine = to_f32<T>(A[(((size_t)b * k_h + i_mine / d) * Tlen + t) * d + i_mine % d]);
    const int m = ids[t];
    if (m < 0 || m >= 32 || !((masks[b] >> m) & 1u)) {             // absent token: zero row
        for (int e = threadIdx.x; e < D; e += blockDim.x) o[e] = from_f32<T>(0.f);
        return;
    }
    for (int j = threadIdx.x; j < k_h; j += blockDim.x) {
        int h = kept_heads[(size_t)b * k_h + j];
        if (h < 0 || h >= Hq) { atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX); h = -1; }
        s_h[j] = h;
    }
    for (int i = threadIdx.x; i < n_a; i += blockDim.x)
        s_a[i] = i == (int)threadIdx.x ? a_mine : to_f32<T>(A[(((size_t)b * k_h + i / d) * Tlen + t) * d + i % d]);
    __syncthreads();
    for (int e = threadIdx.x; e < D; e += blockDim.x) {
        float acc = 0.f;
        for (int j = 0; j < k_h; ++j) {
            const int h = s_h[j];
            if (h < 0) continue;
#pragma unroll 16
            for (int c = 0; c < d; ++c) acc = fmaf(s_a[j * d + c], to_f32<T>(WO[(size_t)(h * d + c) * D + e]), acc);
        }
        o[e] = from_f32<T>(acc);
    }
}

}  // namespace

int launch_project_qkv_generic(sentry_ctx* ctx, const ProjArgs& a, cudaStream_t st) {
    const sentry_proj_desc& d = a.d;
    const unsigned grid = (unsigned)((size_t)d.B * d.T);
    const size_t smem = (size_t)d.D * sizeof(float);
    LaunchScope ls(ctx, KS_PROJ_QKV, st);
    if (d.dtype == SENTRY_F32)
        SENTRY_CUDA_TRY(launch_chained(project_qkv_kernel<float>, dim3(grid), dim3(kProjThreads), smem, st, (const float*)a.X, (const float*)a.WQ, (const float*)a.WK, (const float*)a.WV, a.kept_heads, a.ids, a.masks,
            d.T, d.D, d.Hq, d.Hk, d.d, d.k_h, (float*)a.Q, (float*)a.K, (float*)a.V, a.status));
    else if (d.dtype == SENTRY_F16)
        SENTRY_CUDA_TRY(launch_chained(project_qkv_kernel<__half>, dim3(grid), dim3(kProjThreads), smem, st, (const __half*)a.X, (const __half*)a.WQ, (const __half*)a.WK, (const __half*)a.WV, a.kept_heads, a.ids,
            a.masks, d.T, d.D, d.Hq, d.Hk, d.d, d.k_h, (__half*)a.Q, (__half*)a.K, (__half*)a.V, a.status));
    else
        SENTRY_CUDA_TRY(launch_chained(project_qkv_kernel<__nv_bfloat16>, dim3(grid), dim3(kProjThreads), smem, st, (const __nv_bfloat16*)a.X, (const __nv_bfloat16*)a.WQ, (const __nv_bfloat16*)a.WK,
            (const __nv_bfloat16*)a.WV, a.kept_heads, a.ids, a.masks, d.T, d.D, d.Hq, d.Hk, d.d, d.k_h,
            (__nv_bfloat16*)a.Q, (__nv_bfloat16*)a.K, (__nv_bfloat16*)a.V, a.status));
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}

int launch_project_out_generic(sentry_ctx* ctx, const ProjArgs& a, cudaStream_t st) {
    const sentry_proj_desc& d = a.d;
    const unsigned grid = (unsigned)((size_t)d.B * d.T);
    const size_t smem = (size_t)d.k_h * d.d * sizeof(float);
    LaunchScope ls(ctx, KS_PROJ_OUT, st);
    if (d.dtype == SENTRY_F32)
        SENTRY_CUDA_TRY(launch_chained(project_out_kernel<float>, dim3(grid), dim3(kProjThreads), smem, st, (const float*)a.A, (const float*)a.WO, a.kept_heads, a.ids, a.masks, d.T, d.D, d.Hq, d.d, d.k_h,
            (float*)a.out, a.status));
    else if (d.dtype == SENTRY_F16)
        SENTRY_CUDA_TRY(launch_chained(project_out_kernel<__half>, dim3(grid), dim3(kProjThreads), smem, st, (const __half*)a.A, (const __half*)a.WO, a.kept_heads, a.ids, a.masks, d.T, d.D, d.Hq, d.d, d.k_h,
            (__half*)a.out, a.status));
    else
        SENTRY_CUDA_TRY(launch_chained(project_out_kernel<__nv_bfloat16>, dim3(grid), dim3(kProjThreads), smem, st, (const __nv_bfloat16*)a.A, (const __nv_bfloat16*)a.WO, a.kept_heads, a.ids, a.masks, d.T, d.D, d.Hq, d.d,
            d.k_h, (__nv_bfloat16*)a.out, a.status));
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}
