// SentryGate evaluated on the device (Section 4.2, Eq. 1): for every unit i (attention head or FFN
// channel, the units of all layers concatenated) and every modality mask value s,
//   z_i(s) = zeta_i + gamma_l(i) * f_i(m_s),   g_i(s) = sigmoid(z_i(s)),
//   f_i(m) = w2_i . relu(W1_i m + b1_i) + b2_i        (a two-layer perceptron per unit),
// m_s = the bits of s.  The table of logits z [S, N] is what sentry_gate_select ranks: one row per
// mask value, so the "global threshold over all layers" of Section 4.6 is a top-k over the whole
// concatenated row; layer_counts then says how many of the kept units fall into each layer.
#include "common.cuh"

namespace {

// A block takes 32 units and up to 64 mask values: a lane is a unit, a warp every eighth mask value.  The units' parameters
// pass through shared memory in pieces of `jc` hidden neurons (coalesced reads; rows padded to an odd number of words, so
// that the 32 units of a warp fall on 32 banks), each read once for all mask values.  (One thread per (mask, unit) reading
// its parameters from global memory: 192-byte strides between lanes, 10.4 us at 4096 units x 8 masks x 16 neurons; this
// form 4.)  The few multiply-adds run in fp32 in the order of the definition.
constexpr int kEvalUnits = 32, kEvalMasks = 64, kEvalWords = 8192;

__global__ void __launch_bounds__(256)
gate_eval_kernel(const float* __restrict__ zeta, const float* __restrict__ gamma,
                 const int32_t* __restrict__ layer_offsets, int n_layers, const float* __restrict__ W1,
                 const float* __restrict__ b1, const float* __restrict__ w2, const float* __restrict__ b2,
                 int M, int hidden, int jc, int N, int S, float* __restrict__ logits, float* __restrict__ gates) {
    grid_dependents_start();
    grid_dependency_wait();
    extern __shared__ float s_par[];               // [32][stride]: W1 piece [jc][M] | b1 piece [jc] | w2 piece [jc]
    const int stride = (jc * (M + 2)) | 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int u0 = blockIdx.x * kEvalUnits, nu = min(kEvalUnits, N - u0);
    const int s0 = blockIdx.y * kEvalMasks;
    const int i = u0 + lane;
    const bool live = lane < nu;
    float f[kEvalMasks / 8];
#pragma unroll
    for (int q = 0; q < kEvalMasks / 8; ++q) f[q] = live ? b2[i] : 0.f;
    int l = 0;
    if (live)
        while (l + 1 < n_layers && i >= layer_offsets[l + 1]) ++l;
    const float gam = gamma[l], zet = live ? zeta[i] : 0.f;
    const float* mine = s_par + lane * stride;
    for (int j0 = 0; j0 < hidden; j0 += jc) {
        const int nj = min(jc, hidden - j0);
        __syncthreads();
        if (jc == hidden) {                        // whole units: one contiguous piece, every thread's loads in flight at once
            const float* src = W1 + (size_t)u0 * hidden * M;
            const int hm = hidden * M;
#pragma unroll 8
            for (int e = threadIdx.x; e < nu * hm; e += 256) s_par[(e / hm) * stride + e % hm] = src[e];
#pragma unroll 4
            for (int e = threadIdx.x; e < nu * hidden; e += 256) {
                const int u = e / hidden, j = e % hidden;
                s_par[u * stride + hm + j] = b1[(size_t)u0 * hidden + e];
                s_par[u * stride + hm + hidden + j] = w2[(size_t)u0 * hidden + e];
            }
        } else {
            for (int u = warp; u < nu; u += 8) {   // a warp per unit
                const float* src = W1 + ((size_t)(u0 + u) * hidden + j0) * M;
                float* dst = s_par + u * stride;
                for (int e = lane; e < nj * M; e += 32) dst[e] = src[e];
                for (int e = lane; e < nj; e += 32) {
                    dst[jc * M + e] = b1[(size_t)(u0 + u) * hidden + j0 + e];
                    dst[jc * (M + 1) + e] = w2[(size_t)(u0 + u) * hidden + j0 + e];
                }
            }
        }
        __syncthreads();
        if (!live) continue;
#pragma unroll
        for (int q = 0; q < kEvalMasks / 8; ++q) {
            const int s = s0 + warp + 8 * q;
            if (s >= S) break;
            for (int j = 0; j < nj; ++j) {
                float a = mine[jc * M + j];
                for (int m = 0; m < M; ++m)
                    if ((s >> m) & 1) a += mine[j * M + m];
                f[q] = fmaf(mine[jc * (M + 1) + j], fmaxf(a, 0.f), f[q]);
            }
        }
    }
    if (!live) return;
#pragma unroll
    for (int q = 0; q < kEvalMasks / 8; ++q) {
        const int s = s0 + warp + 8 * q;
        if (s >= S) break;
        const float z = fmaf(gam, f[q], zet);
        logits[(size_t)s * N + i] = z;
        if (gates != nullptr) gates[(size_t)s * N + i] = 1.0f / (1.0f + expf(-z));
    }
}

// kept [n_masks, k] ascending unit indices -> counts [n_masks, n_layers].  A block per list; a warp finds the first
// position not below a layer's offset by a 32-way search (three rounds of memory latency up to 32 K entries where a
// binary search takes up to 15), the counts are the differences.  Layers go through shared memory kCountLayers at a time.
constexpr int kCountLayers = 8192;
__global__ void __launch_bounds__(256)
layer_count_kernel(const int32_t* __restrict__ kept, int n_masks, int k, const int32_t* __restrict__ layer_offsets,
                   int n_layers, int32_t* __restrict__ counts) {
    grid_dependents_start();
    grid_dependency_wait();
    extern __shared__ int s_pos[];                 // [min(n_layers, kCountLayers) + 1]
    const int m = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t* row = kept + (size_t)m * k;
    for (int l0 = 0; l0 < n_layers; l0 += kCountLayers) {
        const int nl = min(n_layers - l0, kCountLayers);
        for (int l = warp; l <= nl; l += 8) {
            const int bound = layer_offsets[l0 + l];
            int lo = 0, hi = k;                    // row[lo - 1] < bound <= row[hi]
            while (lo < hi) {
                const int step = (hi - lo + 31) / 32;
                const int at = lo + step * (lane + 1) - 1;
                const bool below = at < hi && row[at] < bound;
                const int n = __popc(__ballot_sync(0xffffffffu, below));   // probes below the bound: the first n lanes
                hi = min(hi, lo + step * (n + 1) - 1);
                lo += step * n;
                hi = max(hi, lo);
            }
            if (lane == 0) s_pos[l] = lo;
        }
        __syncthreads();
        for (int l = threadIdx.x; l < nl; l += blockDim.x) counts[(size_t)m * n_layers + l0 + l] = s_pos[l + 1] - s_pos[l];
        __syncthreads();
    }
}

}  // namespace

int launch_gate_eval(sentry_ctx* ctx, const float* zeta, const float* gamma, const int32_t* layer_offsets,
                     int n_layers, const float* W1, const float* b1, const float* w2, const float* b2, int M,
                     int hidden, int N, float* logits, float* gates, cudaStream_t st) {
    const int S = 1 << M;
    int jc = kEvalWords / (kEvalUnits * (M + 2));
    if (jc > hidden) jc = hidden;
    const size_t smem = (size_t)kEvalUnits * ((jc * (M + 2)) | 1) * sizeof(float);   // at most 33 KB
    const dim3 grid((unsigned)((N + kEvalUnits - 1) / kEvalUnits), (unsigned)((S + kEvalMasks - 1) / kEvalMasks));
    LaunchScope ls(ctx, KS_GATE_EVAL, st);
    SENTRY_CUDA_TRY(launch_chained(gate_eval_kernel, dim3(grid), dim3(256), smem, st, zeta, gamma, layer_offsets, n_layers, W1, b1, w2, b2, M, hidden, jc, N, S,
                                              logits, gates));
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}

int launch_layer_counts(sentry_ctx* ctx, const int32_t* kept, int n_masks, int k, const int32_t* layer_offsets,
                        int n_layers, int32_t* counts, cudaStream_t st) {
    LaunchScope ls(ctx, KS_GATE_EVAL, st);
    const size_t smem = ((size_t)(n_layers < kCountLayers ? n_layers : kCountLayers) + 1) * sizeof(int);
    SENTRY_CUDA_TRY(launch_chained(layer_count_kernel, dim3(n_masks), dim3(256), smem, st, kept, n_masks, k, layer_offsets, n_layers, counts));
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}
