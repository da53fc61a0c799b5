// SentryGate selection (Section 4.6): per modality-mask row of the score
// table, keep the k best-scoring units; then fan the per-row result out to the
// per-sample masks.  Selection is exact and deterministic: scores are mapped to
// order-preserving integer keys, the k-th key is found by counting against
// candidate thresholds, and the kept indices are compacted in ascending order
// (equal scores: lower index first).
#include "common.cuh"

namespace {

// ------------------------------------------------------------------------------------------
// Rows of up to kGateMaxRegUnits units: a thread holds KPT consecutive keys in registers, and one launch does the
// selection and the fan-out to the samples.
//
// Bound by latency: a row is a few KB, and what takes the time is the chain of block-wide steps.  A counting step costs
// about 270 cycles at 256 threads (warp votes, a barrier, a 56-cycle warp reduction), so a step settles TWO bits of the
// k-th key (three candidate thresholds at once), the search starts at the first bit in which the keys differ and ends as
// soon as exactly k keys lie above a candidate: 6 to 8 steps.  Few threads with several keys each, because the barrier
// of 1024 threads costs 87 cycles and that of 256 costs 39.
// grid (S * sets, y): the y blocks of a row each make the row's selection and serve their share of the samples -- one
// launch whatever the fan-out, where a second launch for large fan-outs cost more than the repeated selection.
struct GateSetDev {
    const float* scores;
    int n_units, k;
    int heads_per_group;
    const uint32_t* masks;
    int n_masks;
    int32_t* kept;
    uint32_t* kv_groups;
};
struct GateSetsDev { GateSetDev set[SENTRY_GATE_MAX_SETS]; };

constexpr int kGateMaxRegUnits = 8192;

template <int KPT>
__global__ void __launch_bounds__(1024)
gate_select_kernel(const __grid_constant__ GateSetsDev sets, int S, unsigned int* status) {
    grid_dependency_wait();
    extern __shared__ int32_t s_list[];            // [k] kept units, ascending
    __shared__ uint32_t s_red[2][3][32];           // per-warp partial results of a counting step, two steps in turn
    __shared__ uint32_t s_bits;
    const GateSetDev& g = sets.set[blockIdx.x / S];
    const int s = (int)(blockIdx.x % S), n = g.n_units, k = g.k;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const float* row = g.scores + (size_t)s * n;
    const int i0 = threadIdx.x * KPT;
    uint32_t key[KPT];
    uint32_t hi = 0u, lo = 0xffffffffu;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
        // padding ranks with NaN, below every number; it is kept out of the list by its index
        key[j] = i0 + j < n ? sentry_order_key(__ldg(row + i0 + j)) : 0u;
    }
#pragma unroll
    for (int j = 0; j < KPT; ++j)
        if (i0 + j < n) { hi = max(hi, key[j]); lo = min(lo, key[j]); }
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_min_sync(0xffffffffu, lo);
    if (lane == 0) { s_red[0][0][warp] = hi; s_red[0][1][warp] = lo; }
    if (threadIdx.x == 0) s_bits = 0u;
    __syncthreads();
    hi = __reduce_max_sync(0xffffffffu, lane < nw ? s_red[0][0][lane] : 0u);
    lo = __reduce_min_sync(0xffffffffu, lane < nw ? s_red[0][1][lane] : 0xffffffffu);

    uint32_t t = lo;
    bool cut = k == n;                             // exactly k units have keys >= t
    int above = 0;                                 // units with keys >= the next candidate above t's range
    if (!cut && hi != lo) {
        int b = (31 - __clz((int)(hi ^ lo))) | 1;  // digits of two bits, aligned
        t = b == 31 ? 0u : hi & ~((2u << b) - 1u);
        int buf = 1;
#pragma unroll 1
        for (b -= 1; b >= 0 && !cut; b -= 2, buf ^= 1) {
            const uint32_t c1 = t + (1u << b), c2 = t + (2u << b), c3 = t + (3u << b);
            uint32_t n1 = 0u, n2 = 0u, n3 = 0u;
#pragma unroll
            for (int j = 0; j < KPT; ++j) {
                n1 += __popc(__ballot_sync(0xffffffffu, key[j] >= c1));
                n2 += __popc(__ballot_sync(0xffffffffu, key[j] >= c2));
                n3 += __popc(__ballot_sync(0xffffffffu, key[j] >= c3));
            }
            if (lane == 0) { s_red[buf][0][warp] = n1; s_red[buf][1][warp] = n2; s_red[buf][2][warp] = n3; }
            __syncthreads();                       // (the other buffer's readers are past the barrier before)
            const int k1 = (int)__reduce_add_sync(0xffffffffu, lane < nw ? s_red[buf][0][lane] : 0u);
            const int k2 = (int)__reduce_add_sync(0xffffffffu, lane < nw ? s_red[buf][1][lane] : 0u);
            const int k3 = (int)__reduce_add_sync(0xffffffffu, lane < nw ? s_red[buf][2][lane] : 0u);
            if (k3 >= k) { t = c3; cut = k3 == k; }
            else if (k2 >= k) { t = c2; cut = k2 == k; above = k3; }
            else if (k1 >= k) { t = c1; cut = k1 == k; above = k2; }
            else above = k1;
        }
        __syncthreads();
    } else {
        __syncthreads();
    }
    // ordered compaction.  cut: everything >= t (t may be 0 only with k == n).  Otherwise t is the k-th key itself: all
    // keys above it (`above` of them) and, in index order, as many of the equal ones as are wanted
    const int need_eq = cut ? 0x7fffffff : k - above;
    uint32_t mine = 0u;                            // keys above t: low half, equal to t: high half
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
        const bool in = i0 + j < n;
        mine += (in && key[j] > t ? 1u : 0u) + (in && key[j] == t ? 65536u : 0u);
    }
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) s_red[0][2][warp] = incl;
    __syncthreads();
    const uint32_t warps_before = __reduce_add_sync(0xffffffffu, lane < warp ? s_red[0][2][lane] : 0u);
    const uint32_t before = warps_before + incl - mine;
    int gt_n = (int)(before & 0xffffu), eq_n = (int)(before >> 16);
    uint32_t bits = 0u;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
        const bool in = i0 + j < n, gt = in && key[j] > t, eq = in && key[j] == t;
        if (gt || (eq && eq_n < need_eq)) {
            s_list[gt_n + min(eq_n, need_eq)] = i0 + j;
            if (g.kv_groups != nullptr) bits |= 1u << ((i0 + j) / g.heads_per_group);
        }
        gt_n += gt;
        eq_n += eq;
    }
    if (g.kv_groups != nullptr && bits) atomicOr(&s_bits, bits);
    __syncthreads();

    // fan-out over this block's share of the samples
    const int per = (g.n_masks + (int)gridDim.y - 1) / (int)gridDim.y;
    const int m_end = min(g.n_masks, ((int)blockIdx.y + 1) * per);
    if (k <= 16) {                                 // short lists (heads): a thread per sample
        for (int m = (int)blockIdx.y * per + threadIdx.x; m < m_end; m += blockDim.x) {
            const uint32_t ms = g.masks[m];
            if (ms == (uint32_t)s) {
                for (int j = 0; j < k; ++j) g.kept[(size_t)m * k + j] = s_list[j];
                if (g.kv_groups != nullptr) g.kv_groups[m] = s_bits;
            } else if (s == 0 && ms >= (uint32_t)S) {
                atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
            }
        }
        return;
    }
    for (int m0 = (int)blockIdx.y * per; m0 < m_end; m0 += 32) {   // longer ones: the block copies the list to each match
        const uint32_t ms = m0 + lane < m_end ? g.masks[m0 + lane] : 0xfffffffeu;
        if (s == 0 && warp == 0 && m0 + lane < m_end && ms >= (uint32_t)S) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
        unsigned hits = __ballot_sync(0xffffffffu, m0 + lane < m_end && ms == (uint32_t)s);
        while (hits) {
            const int m = m0 + __ffs(hits) - 1;
            hits &= hits - 1;
            for (int j = threadIdx.x; j < k; j += blockDim.x) g.kept[(size_t)m * k + j] = s_list[j];
            if (g.kv_groups != nullptr && threadIdx.x == 0) g.kv_groups[m] = s_bits;
        }
    }
}

// Launch of the register form: keys per thread and threads from the longest row, blocks per row from the fan-out.
int launch_gate_reg(int S, const sentry_gate_set* sets, int n_sets, unsigned int* status, int sm_count,
                    cudaStream_t st) {
    GateSetsDev dev = {};
    int n_max = 1, k_max = 1, m_max = 1;
    long long out_max = 1;
    for (int i = 0; i < n_sets; ++i) {
        const sentry_gate_set& g = sets[i];
        dev.set[i] = {g.scores, g.n_units, g.k, g.heads_per_group > 0 ? g.heads_per_group : 1, g.masks, g.n_masks, g.kept, g.kv_groups};
        if (g.n_units > n_max) n_max = g.n_units;
        if (g.k > k_max) k_max = g.k;
        if (g.n_masks > m_max) m_max = g.n_masks;
        if ((long long)g.n_masks * g.k > out_max) out_max = (long long)g.n_masks * g.k;
    }
    // a share of 4096 list entries and 512 samples per block, as long as the blocks of all rows together about fill the GPU once
    long long y = (out_max / S + 4095) / 4096;
    if (y < (m_max + 511) / 512) y = (m_max + 511) / 512;
    const long long most = (sm_count + S * n_sets - 1) / (S * n_sets);
    if (y > most) y = most;
    if (y < 1) y = 1;
    const dim3 grid((unsigned)(S * n_sets), (unsigned)y);
    const size_t smem = (size_t)k_max * sizeof(int32_t);
    auto threads_for = [&](int kpt) { return ((n_max + kpt - 1) / kpt + 31) / 32 * 32; };
    if (n_max <= 256) {
        const int th = n_max <= 64 ? (out_max >= 1024 ? 256 : 64) : threads_for(1);
        SENTRY_CUDA_TRY(launch_chained(gate_select_kernel<1>, dim3(grid), dim3(th), smem, st, dev, S, status));
    } else if (n_max <= 1024) {
        SENTRY_CUDA_TRY(launch_chained(gate_select_kernel<4>, dim3(grid), dim3(threads_for(4)), smem, st, dev, S, status));
    } else {
        SENTRY_CUDA_TRY(launch_chained(gate_select_kernel<8>, dim3(grid), dim3(threads_for(8)), smem, st, dev, S, status));
    }
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}


constexpr int kGateMaxThreads = 1024;

// ------------------------------------------------------------------------------------------
// Longer rows: keys in shared memory, the rows to scratch, a second launch fans them out.
// One block per score-table row s: rows[s, 0..k) and groups[s].
__global__ void __launch_bounds__(kGateMaxThreads)
gate_rows_kernel(const float* __restrict__ scores, int n_units, int k, int32_t* __restrict__ rows,
                 uint32_t* __restrict__ groups, int heads_per_group) {
    extern __shared__ uint32_t s_keys[];
    __shared__ int red[66];
    __shared__ uint32_t s_bits;
    const int s = blockIdx.x;
    const float* row = scores + (size_t)s * n_units;
    for (int i = threadIdx.x; i < n_units; i += blockDim.x) s_keys[i] = sentry_order_key(row[i]);
    if (threadIdx.x == 0) s_bits = 0u;
    __syncthreads();
    int32_t* out = rows + (size_t)s * k;
    block_select_topk(s_keys, n_units, k, out, nullptr, red);
    if (groups != nullptr) {
        uint32_t bits = 0u;
        for (int i = threadIdx.x; i < k; i += blockDim.x) bits |= 1u << (out[i] / heads_per_group);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) bits |= __shfl_xor_sync(0xffffffffu, bits, o);
        if ((threadIdx.x & 31) == 0 && bits) atomicOr(&s_bits, bits);
        __syncthreads();
        if (threadIdx.x == 0) groups[s] = s_bits;
    }
}

// kept[m, :] = rows[masks[m], :]  (and kv_groups[m] = groups[masks[m]]).
__global__ void gate_expand_kernel(const int32_t* __restrict__ rows,
                                   const uint32_t* __restrict__ groups,
                                   const uint32_t* __restrict__ masks, int S, int n_masks, int k,
                                   int32_t* __restrict__ kept, uint32_t* __restrict__ kv_groups,
                                   unsigned int* status) {
    const size_t total = (size_t)n_masks * k;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        const int m = (int)(i / k), j = (int)(i % k);
        const uint32_t s = masks[m];
        if (s >= (uint32_t)S) {
            if (j == 0) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
            continue;
        }
        kept[i] = rows[(size_t)s * k + j];
        if (j == 0 && kv_groups != nullptr) kv_groups[m] = groups[s];
    }
}

}  // namespace

int launch_gate_select(sentry_ctx* ctx, const float* scores, int S, int n_units,
                       const uint32_t* masks, int n_masks, int k, int32_t* kept,
                       uint32_t* kv_groups, int heads_per_group, int32_t* ws_rows,
                       uint32_t* ws_groups, cudaStream_t st) {
    if (n_units <= kGateMaxRegUnits) {
        const sentry_gate_set g = {scores, n_units, k, masks, n_masks, kept, kv_groups, heads_per_group};
        LaunchScope ls(ctx, KS_GATE_ROWS, st);
        return launch_gate_reg(S, &g, 1, ctx->d_status, ctx->sm_count, st);
    }
    const size_t smem = (size_t)n_units * sizeof(uint32_t);
    if (smem > 48 * 1024)
        SENTRY_CUDA_TRY(cudaFuncSetAttribute(gate_rows_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const size_t total = (size_t)n_masks * k;
    {
        LaunchScope ls(ctx, KS_GATE_ROWS, st);
        gate_rows_kernel<<<S, kGateMaxThreads, smem, st>>>(scores, n_units, k, ws_rows, kv_groups ? ws_groups : nullptr,
                                                           heads_per_group > 0 ? heads_per_group : 1);
    }
    SENTRY_CUDA_TRY(cudaGetLastError());
    int blocks = (int)((total + 255) / 256);
    const int cap = ctx->sm_count * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    {
        LaunchScope ls(ctx, KS_GATE_EXPAND, st);
        gate_expand_kernel<<<blocks, 256, 0, st>>>(ws_rows, ws_groups, masks, S, n_masks, k, kept,
                                                   kv_groups, ctx->d_status);
    }
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}

// All sets in one launch; with a row too long for the register form, set after set.
int launch_gate_select_multi(sentry_ctx* ctx, int S, const sentry_gate_set* sets, int n_sets, int32_t* const* ws_rows,
                             uint32_t* const* ws_groups, cudaStream_t st) {
    bool all_short = true;
    for (int i = 0; i < n_sets; ++i) all_short = all_short && sets[i].n_units <= kGateMaxRegUnits;
    if (all_short) {
        LaunchScope ls(ctx, KS_GATE_ROWS, st);
        return launch_gate_reg(S, sets, n_sets, ctx->d_status, ctx->sm_count, st);
    }
    for (int i = 0; i < n_sets; ++i) {
        const sentry_gate_set& g = sets[i];
        if (g.n_masks == 0) continue;
        const int rc = launch_gate_select(ctx, g.scores, S, g.n_units, g.masks, g.n_masks, g.k, g.kept, g.kv_groups,
                                          g.heads_per_group, ws_rows[i], ws_groups[i], st);
        if (rc != SENTRY_OK) return rc;
    }
    return SENTRY_OK;
}

// ------------------------------------------------------------------------------------------
// Allocation-free variant of the gate selection.
//
// Its scratch (the per-score-row result that the fan-out kernel reads, the per-row KV-group
// bitmaps and a status word) lives in one file-scope device array instead of a workspace, so
// a caller that is not allowed to call cudaMalloc -- code running inside another runtime's
// memory pool, or an embedding that fixes its device-memory budget at start-up -- can still
// run the selection.  The array is part of the library image: every GPU that loads the
// library holds these 256 KB until the process exits.
//
// In host code `g_gate_scratch` is only a handle for the symbol, not a device address;
// the address a kernel can use comes from cudaGetSymbolAddress, asked once per device with
// that device current (static_scratch_of below).
#include <mutex>

namespace {

static __device__ __align__(256) unsigned char g_gate_scratch[SENTRY_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
constexpr size_t kStaticHeader = 256;  // status word, padded so the tables stay 256-byte aligned

struct StaticDevice {
    unsigned char* scratch = nullptr;  // device address of g_gate_scratch on this device
    int sm_count = 0;
};
StaticDevice g_static_dev[kMaxDevices];
std::mutex g_static_mu;

// Device address of the scratch array on `device` (which must be current).  The first call per
// device asks the runtime for it; later calls only read the cached value.
int static_scratch_of(int device, StaticDevice* out) {
    std::lock_guard<std::mutex> lock(g_static_mu);
    StaticDevice& sd = g_static_dev[device];
    if (sd.scratch == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_gate_scratch) != cudaSuccess || p == nullptr) {
            cudaGetLastError();
            return SENTRY_ERR_CUDA;
        }
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || sms < 1)
            return SENTRY_ERR_CUDA;
        sd.sm_count = sms;
        sd.scratch = static_cast<unsigned char*>(p);
    }
    *out = sd;
    return SENTRY_OK;
}

}  // namespace

extern "C" int sentry_gate_select_static(int device, const float* scores, int S, int n_units,
                                         const uint32_t* masks, int n_masks, int k, int32_t* kept,
                                         uint32_t* kv_groups, int heads_per_group,
                                         uint32_t* status, void* stream) {
    if (scores == nullptr || masks == nullptr || kept == nullptr) return SENTRY_ERR_INVALID_ARG;
    if (((uintptr_t)scores | (uintptr_t)masks | (uintptr_t)kept | (uintptr_t)kv_groups |
         (uintptr_t)status) % 4 != 0)
        return SENTRY_ERR_INVALID_ARG;
    if (device < 0 || device >= kMaxDevices) return SENTRY_ERR_INVALID_ARG;
    if (S < 1 || n_units < 1 || n_masks < 0 || k < 1 || k > n_units) return SENTRY_ERR_BAD_SHAPE;
    if (kv_groups != nullptr) {
        if (heads_per_group < 1) return SENTRY_ERR_INVALID_ARG;
        if ((n_units + heads_per_group - 1) / heads_per_group > 32) return SENTRY_ERR_BAD_SHAPE;
    }
    // the sort keys of one score row must fit the default shared-memory window
    if ((size_t)n_units * sizeof(uint32_t) > 48 * 1024) return SENTRY_ERR_UNSUPPORTED;
    // rows [S,k] i32 and groups [S] u32 must fit the static array
    const size_t rows_bytes = align_up((size_t)S * k * sizeof(int32_t), 256);
    const size_t groups_bytes = (size_t)S * sizeof(uint32_t);
    if (kStaticHeader + rows_bytes + groups_bytes > (size_t)SENTRY_STATIC_SCRATCH_BYTES)
        return SENTRY_ERR_WORKSPACE;
    if (n_masks == 0) return SENTRY_OK;

    SENTRY_ON_DEVICE(device);
    StaticDevice sd;
    int rc = static_scratch_of(device, &sd);
    if (rc != SENTRY_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    unsigned int* own_status = reinterpret_cast<unsigned int*>(sd.scratch);
    int32_t* rows = reinterpret_cast<int32_t*>(sd.scratch + kStaticHeader);
    uint32_t* groups = reinterpret_cast<uint32_t*>(sd.scratch + kStaticHeader + rows_bytes);
    if (n_units <= kGateMaxRegUnits) {   // no scratch wanted
        const sentry_gate_set g = {scores, n_units, k, masks, n_masks, kept, kv_groups, heads_per_group};
        return launch_gate_reg(S, &g, 1, status != nullptr ? status : own_status, sd.sm_count, st);
    }
    // The array keeps whatever the previous call left.  rows/groups are rewritten in full for
    // all S score rows before the fan-out reads them; only the status word must start at zero.
    SENTRY_CUDA_TRY(cudaMemsetAsync(own_status, 0, sizeof(unsigned int), st));
    gate_rows_kernel<<<S, kGateMaxThreads, (size_t)n_units * sizeof(uint32_t), st>>>(
        scores, n_units, k, rows, kv_groups ? groups : nullptr, heads_per_group > 0 ? heads_per_group : 1);
    SENTRY_CUDA_TRY(cudaGetLastError());
    const size_t total = (size_t)n_masks * k;
    int blocks = (int)((total + 255) / 256);
    if (blocks > sd.sm_count * 8) blocks = sd.sm_count * 8;
    if (blocks < 1) blocks = 1;
    gate_expand_kernel<<<blocks, 256, 0, st>>>(rows, groups, masks, S, n_masks, k, kept, kv_groups,
                                               status != nullptr ? status : own_status);
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}
