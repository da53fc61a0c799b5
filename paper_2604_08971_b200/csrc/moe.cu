// Sparse-MoE block with expert-internal channel pruning (Section 4.6): the routing (which experts a
// token goes to, with which weights) is given and untouched; every expert e runs the compacted pair
// GELU(x W1_e[:, N_e]) W2_e[N_e, :] on the tokens routed to it, and a token's output is the
// weighted sum over its routing slots.
//
// On the device this is the channel-compacted FFN with one kept-channel list AND one weight pair
// per expert:  the (token, slot) pairs are regrouped by expert into the same row plan the dense FFN
// uses (list = expert), with a second row table that sends each result to its own (token, slot)
// row of a staging buffer; the fused-pair kernels run unchanged on that plan; a last kernel forms
// the weighted sum per token in slot order (fp32 accumulation, no atomics on data, so the result
// does not depend on how the rows were grouped).
#include "ffn_plan.cuh"

namespace {

constexpr int kPlanThreads = 256;

// The plan of a large call in two launches.  A block owns a contiguous run of `per_block` slots (a multiple of 2048, eight per
// thread and round).  Count: block b writes its slots per expert to counts[b][E].  Scatter: every block adds up the counts of
// all blocks for itself -- the experts' row ranges, and in them its own first rows -- and then hands out positions from shared
// memory; block 0 leaves list_row0 and tile_start.  No zeroing, no global atomics, no launch of one block in between.
// Bound by latency: 65 536 slots, 8 experts, the routed block 60.8 -> 54.9 us where it was a memset and three launches.
// Slot with id -1: not routed (skipped).  Any other id outside [0, E): status bit, skipped.
constexpr int kRoundSlots = kPlanThreads * 8;
__global__ void __launch_bounds__(kPlanThreads)
moe_count_kernel(const int32_t* __restrict__ expert_ids, long long n_slots, long long per_block, int E,
                 int32_t* __restrict__ counts, unsigned int* status) {
    grid_dependents_start();
    grid_dependency_wait();
    extern __shared__ int s_cnt[];   // [E]
    const int lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < E; e += kPlanThreads) s_cnt[e] = 0;
    __syncthreads();
    const long long begin = (long long)blockIdx.x * per_block, end = min(n_slots, begin + per_block);
    bool bad = false;
    for (long long i0 = begin; i0 < end; i0 += kRoundSlots) {
        int ev[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const long long i = i0 + (long long)j * kPlanThreads + threadIdx.x;
            ev[j] = i < end ? __ldg(expert_ids + i) : -1;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            int e = ev[j];
            if (e < -1 || e >= E) { bad = true; e = -1; }
            // one shared-memory atomic per (warp, expert)
            const unsigned peers = __match_any_sync(0xffffffffu, e);
            if (e >= 0 && lane == __ffs(peers) - 1) atomicAdd(&s_cnt[e], __popc(peers));
        }
    }
    if (bad) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
    __syncthreads();
    for (int e = threadIdx.x; e < E; e += kPlanThreads) counts[(size_t)blockIdx.x * E + e] = s_cnt[e];
}

__global__ void __launch_bounds__(kPlanThreads)
moe_scatter_kernel(const int32_t* __restrict__ expert_ids, long long n_slots, long long per_block, int E, int top_k,
                   int tile_rows, const int32_t* __restrict__ counts, FfnPlan plan) {
    grid_dependents_start();
    extern __shared__ int s_int[];
    int* s_cnt = s_int;        // [E] slots per expert, all blocks
    int* s_cur = s_int + E;    // [E] of the blocks before this one; then the next free row of the expert
    const int lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < 2 * E; e += kPlanThreads) s_int[e] = 0;
    grid_dependency_wait();
    __syncthreads();
    const int mine = (int)blockIdx.x * E, all = (int)gridDim.x * E;
#pragma unroll 4
    for (int i = threadIdx.x; i < all; i += kPlanThreads) {
        const int v = counts[i], e = i % E;
        if (v > 0) {
            atomicAdd(&s_cnt[e], v);
            if (i < mine) atomicAdd(&s_cur[e], v);
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {   // exclusive prefix sums over the experts, 32 at a time
        int row0 = 0, tile0 = 0;
        for (int e0 = 0; e0 < E; e0 += 32) {
            const int e = e0 + lane;
            const int c = e < E ? s_cnt[e] : 0;
            const int t = (c + tile_rows - 1) / tile_rows;
            int ic = c, it = t;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int vc = __shfl_up_sync(0xffffffffu, ic, o), vt = __shfl_up_sync(0xffffffffu, it, o);
                if (lane >= o) { ic += vc; it += vt; }
            }
            if (e < E) {
                s_cur[e] += row0 + ic - c;
                if (blockIdx.x == 0) {
                    plan.list_row0[e] = row0 + ic - c;
                    plan.tile_start[e] = tile0 + it - t;
                }
            }
            row0 += __shfl_sync(0xffffffffu, ic, 31);
            tile0 += __shfl_sync(0xffffffffu, it, 31);
        }
        if (blockIdx.x == 0 && lane == 0) { plan.list_row0[E] = row0; plan.tile_start[E] = tile0; }
    }
    __syncthreads();
    const long long begin = (long long)blockIdx.x * per_block, end = min(n_slots, begin + per_block);
    for (long long i0 = begin; i0 < end; i0 += kRoundSlots) {
        int ev[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const long long i = i0 + (long long)j * kPlanThreads + threadIdx.x;
            ev[j] = i < end ? __ldg(expert_ids + i) : -1;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const long long i = i0 + (long long)j * kPlanThreads + threadIdx.x;
            const int e = ev[j] < -1 || ev[j] >= E ? -1 : ev[j];
            const unsigned peers = __match_any_sync(0xffffffffu, e);
            const int leader = __ffs(peers) - 1;
            int base = 0;
            if (e >= 0 && lane == leader) base = atomicAdd(&s_cur[e], __popc(peers));
            const int pos = __shfl_sync(0xffffffffu, base, leader) + __popc(peers & ((1u << lane) - 1u));
            if (e >= 0) {
                plan.rowidx[pos] = (int32_t)(i / top_k);   // row of X: the token
                plan.rowout[pos] = (int32_t)i;             // row of the staging buffer: (token, slot)
            }
        }
    }
}

// The whole plan in ONE launch by one block, for small calls (latency: one launch instead of two): count per expert in
// shared memory, prefix sums, then a second walk that hands out the positions (one shared-memory atomic per warp and
// expert in both walks).
constexpr int kPlanOneThreads = 1024;
constexpr long long kPlanOneMaxSlots = 8192;   // one round of the block; beyond it one SM is the slower way (65 536 slots: 53 us)
__global__ void __launch_bounds__(kPlanOneThreads)
moe_plan_one_kernel(const int32_t* __restrict__ expert_ids, int n_slots, int E, int top_k, int tile_rows,
                    FfnPlan plan, unsigned int* status) {
    grid_dependents_start();
    grid_dependency_wait();
    extern __shared__ int s_int[];
    int* s_cnt = s_int;          // [E] slots per expert
    int* s_cur = s_int + E;      // [E] next free row of the expert
    const int lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < E; e += blockDim.x) s_cnt[e] = 0;
    __syncthreads();
    bool bad = false;
    const int per_round = (int)blockDim.x * 8;   // eight ids per thread are requested together
    for (int i0 = 0; i0 < n_slots; i0 += per_round) {
        int ev[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int i = i0 + j * (int)blockDim.x + (int)threadIdx.x;
            ev[j] = i < n_slots ? __ldg(expert_ids + i) : -1;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            int e = ev[j];
            if (e < -1 || e >= E) { bad = true; e = -1; }
            const unsigned peers = __match_any_sync(0xffffffffu, e);
            if (e >= 0 && lane == __ffs(peers) - 1) atomicAdd(&s_cnt[e], __popc(peers));
        }
    }
    if (bad) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
    __syncthreads();
    if (threadIdx.x < 32) {   // exclusive prefix sums over the experts, 32 at a time
        int row0 = 0, tile0 = 0;
        for (int e0 = 0; e0 < E; e0 += 32) {
            const int e = e0 + lane;
            const int c = e < E ? s_cnt[e] : 0;
            const int t = (c + tile_rows - 1) / tile_rows;
            int ic = c, it = t;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int vc = __shfl_up_sync(0xffffffffu, ic, o), vt = __shfl_up_sync(0xffffffffu, it, o);
                if (lane >= o) { ic += vc; it += vt; }
            }
            if (e < E) {
                plan.list_row0[e] = row0 + ic - c;
                plan.tile_start[e] = tile0 + it - t;
                s_cur[e] = row0 + ic - c;
            }
            row0 += __shfl_sync(0xffffffffu, ic, 31);
            tile0 += __shfl_sync(0xffffffffu, it, 31);
        }
        if (lane == 0) { plan.list_row0[E] = row0; plan.tile_start[E] = tile0; }
    }
    __syncthreads();
    for (int i0 = 0; i0 < n_slots; i0 += per_round) {
        int ev[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int i = i0 + j * (int)blockDim.x + (int)threadIdx.x;
            ev[j] = i < n_slots ? __ldg(expert_ids + i) : -1;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int i = i0 + j * (int)blockDim.x + (int)threadIdx.x;
            int e = ev[j];
            if (e < -1 || e >= E) e = -1;
            const unsigned peers = __match_any_sync(0xffffffffu, e);
            const int leader = __ffs(peers) - 1;
            int base = 0;
            if (e >= 0 && lane == leader) base = atomicAdd(&s_cur[e], __popc(peers));
            const int pos = __shfl_sync(0xffffffffu, base, leader) + __popc(peers & ((1u << lane) - 1u));
            if (e >= 0) {
                plan.rowidx[pos] = i / top_k;   // row of X: the token
                plan.rowout[pos] = i;           // row of the staging buffer: (token, slot)
            }
        }
    }
}

template <typename T> struct Vec16;
template <> struct Vec16<float> { static constexpr int N = 4; };
template <> struct Vec16<__nv_bfloat16> { static constexpr int N = 8; };
template <> struct Vec16<__half> { static constexpr int N = 8; };

__device__ __forceinline__ void unpack16(const uint4& v, float (&f)[4]) {
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y);
    f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
}
__device__ __forceinline__ void unpack16(const uint4& v, float (&f)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        f[2 * i] = __uint_as_float(w[i] << 16);
        f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
}
__device__ __forceinline__ uint4 pack16(const float (&f)[4]) {
    return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
}
__device__ __forceinline__ uint4 pack16(const float (&f)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 p = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
        w[i] = *reinterpret_cast<const uint32_t*>(&p);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ void unpack16_half(const uint4& v, float (&f)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 p = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
        f[2 * i] = p.x;
        f[2 * i + 1] = p.y;
    }
}
__device__ __forceinline__ uint4 pack16_half(const float (&f)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __half2 p = __floats2half2_rn(f[2 * i], f[2 * i + 1]);
        w[i] = *reinterpret_cast<const uint32_t*>(&p);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// y_t = sum_j weight[t][j] * staged[t*top_k + j]  over the routed slots, 16 bytes per thread.
template <typename T>
__global__ void __launch_bounds__(256)
moe_combine_kernel(const uint4* __restrict__ staged, const int32_t* __restrict__ expert_ids,
                   const float* __restrict__ weights, long long N, int vpr, int E, int top_k,
                   uint4* __restrict__ Y) {
    grid_dependents_start();
    grid_dependency_wait();
    constexpr int NV = Vec16<T>::N;
    constexpr bool IS_BF16 = sizeof(T) == 2 && Vec16<T>::N == 8 && __is_same(T, __nv_bfloat16);
    const long long total = N * vpr;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long t = i / vpr;
        const int v = (int)(i % vpr);
        float acc[NV];
#pragma unroll
        for (int c = 0; c < NV; ++c) acc[c] = 0.f;
        // four slots at a time: ids, weights and staged rows are requested together (a staged row is
        // read whether or not its slot is routed -- the buffer is there -- and dropped afterwards, so
        // that the row does not wait for the id); the sum runs in slot order
        for (int j0 = 0; j0 < top_k; j0 += 4) {
            int e[4];
            float g[4];
            uint4 raw[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = j0 + u;
                e[u] = -1;
                if (j < top_k) {
                    e[u] = __ldg(expert_ids + t * top_k + j);
                    g[u] = __ldg(weights + t * top_k + j);
                    raw[u] = __ldg(&staged[(t * top_k + j) * vpr + v]);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (e[u] < 0 || e[u] >= E) continue;
                float f[NV];
                if constexpr (sizeof(T) == 2 && !IS_BF16) unpack16_half(raw[u], f);
                else unpack16(raw[u], f);
#pragma unroll
                for (int c = 0; c < NV; ++c) acc[c] = fmaf(g[u], f[c], acc[c]);
            }
        }
        if constexpr (sizeof(T) == 2 && !IS_BF16) Y[i] = pack16_half(acc);
        else Y[i] = pack16(acc);
    }
}

struct MoeWs {
    FfnPlan plan;
    int32_t* counts;   // [plan blocks][E]
    void* staged;
    void* packed;
    void* hidden;
    bool ok;
    size_t used;
};

sentry_ffn_desc as_ffn_desc(const sentry_moe_desc& m) {
    sentry_ffn_desc d;
    d.B = m.N;
    d.T = m.top_k;   // the plan has N * top_k rows
    d.D = m.D; d.F = m.F; d.k_c = m.k_c; d.n_lists = m.E; d.dtype = m.dtype;
    return d;
}

long long tiles_bound(const sentry_moe_desc& m) {
    const int tile_rows = ffn_tile_rows(as_ffn_desc(m));
    return ((long long)m.N * m.top_k + tile_rows - 1) / tile_rows + m.E;
}

// Blocks of the two-launch plan: 2048 slots each, while the counts that every block adds up stay a few thousand.
int plan_blocks(const sentry_moe_desc& m) {
    const long long want = ((long long)m.N * m.top_k + kRoundSlots - 1) / kRoundSlots;
    const long long most = 16384 / m.E < 16 ? 16 : (m.E < 64 ? 256 : 16384 / m.E);
    return (int)(want < most ? want : most);
}

MoeWs carve(const sentry_moe_desc& m, void* ws, size_t bytes, bool with_weights) {
    WsAlloc a(ws, bytes);
    MoeWs w;
    const size_t slots = (size_t)m.N * m.top_k;
    const size_t esz = m.dtype == SENTRY_F32 ? 4 : 2;
    w.plan.sample_row0 = a.take<int32_t>(1);
    w.plan.list_row0 = a.take<int32_t>((size_t)m.E + 1);
    w.plan.tile_start = a.take<int32_t>((size_t)m.E + 1);
    w.plan.rowidx = a.take<int32_t>(slots);
    w.plan.rowout = a.take<int32_t>(slots);
    w.plan.zero_ids = nullptr;
    w.plan.zero_masks = nullptr;
    w.plan.n_rows = 0;
    w.plan.Tlen = 1;
    w.counts = a.take<int32_t>((size_t)plan_blocks(m) * m.E);
    w.staged = a.take<uint8_t>(slots * m.D * esz);
    w.packed = with_weights ? a.take<uint8_t>(ffn_packed_bytes(as_ffn_desc(m))) : nullptr;
    w.hidden = a.take<uint8_t>(ffn_hidden_bytes(as_ffn_desc(m), tiles_bound(m)));
    w.ok = a.ok;
    w.used = a.off;
    return w;
}

}  // namespace

size_t moe_workspace_bytes(const sentry_moe_desc& m) { return carve(m, nullptr, 0, true).used + 256; }
size_t moe_packed_bytes(const sentry_moe_desc& m) { return ffn_packed_bytes(as_ffn_desc(m)); }

int launch_moe_prepack(sentry_ctx* ctx, const MoeArgs& m, void* packed, cudaStream_t st) {
    FfnArgs a = {};
    a.d = as_ffn_desc(m.d);
    a.W1 = m.W1; a.W2 = m.W2;
    a.kept = m.kept;
    a.w_stride = (size_t)m.d.D * m.d.F;
    a.status = m.status;
    return launch_ffn_prepack(ctx, a, packed, st);
}

int launch_moe_ffn(sentry_ctx* ctx, const MoeArgs& m, void* ws, size_t ws_bytes, const void* packed,
                   cudaStream_t st) {
    const sentry_moe_desc& d = m.d;
    MoeWs w = carve(d, ws, ws_bytes, packed == nullptr);
    if (!w.ok) return SENTRY_ERR_WORKSPACE;
    const sentry_ffn_desc fd = as_ffn_desc(d);
    const int tile_rows = ffn_tile_rows(fd);
    const long long slots = (long long)d.N * d.top_k;
    const size_t route_smem = (size_t)2 * d.E * sizeof(int);

    if (packed == nullptr) {
        int rc = launch_moe_prepack(ctx, m, w.packed, st);
        if (rc != SENTRY_OK) return rc;
        packed = w.packed;
    }
    if (slots <= kPlanOneMaxSlots) {
        LaunchScope ls(ctx, KS_MOE_PLAN, st);
        SENTRY_CUDA_TRY(launch_chained(moe_plan_one_kernel, dim3(1), dim3(kPlanOneThreads), route_smem, st, m.expert_ids, (int)slots, d.E, d.top_k, tile_rows,
                                                                    w.plan, m.status));
    } else {
        const int blocks = plan_blocks(d);
        const long long per = ((slots + blocks - 1) / blocks + kRoundSlots - 1) / kRoundSlots * kRoundSlots;
        LaunchScope ls(ctx, KS_MOE_PLAN, st, 2);
        SENTRY_CUDA_TRY(launch_chained(moe_count_kernel, dim3(blocks), dim3(kPlanThreads), route_smem / 2, st, m.expert_ids, slots, per,
                                       d.E, w.counts, m.status));
        SENTRY_CUDA_TRY(launch_chained(moe_scatter_kernel, dim3(blocks), dim3(kPlanThreads), route_smem, st, m.expert_ids, slots, per,
                                       d.E, d.top_k, tile_rows, w.counts, w.plan));
    }
    SENTRY_CUDA_TRY(cudaGetLastError());

    FfnArgs a = {};
    a.d = fd;
    a.X = m.X;
    a.Y = w.staged;
    a.status = m.status;
    const int kc_pad = ffn_kc_pad(fd);
    const int max_tiles = (int)tiles_bound(d);
    void* w1p = const_cast<void*>(packed);
    void* w2p = (uint8_t*)w1p + ffn_packed_bytes(fd) / 2;
    int rc = launch_ffn_main(ctx, a, w.plan, w1p, w2p, kc_pad, max_tiles, w.hidden, st);
    if (rc != SENTRY_OK) return rc;

    {
        const int esz = d.dtype == SENTRY_F32 ? 4 : 2;
        const int vpr = d.D * esz / 16;
        const long long total = (long long)d.N * vpr;
        long long blocks = (total + 255) / 256;
        const long long cap = (long long)ctx->sm_count * 16;
        if (blocks > cap) blocks = cap;
        LaunchScope ls(ctx, KS_MOE_COMBINE, st);
        if (d.dtype == SENTRY_F32)
            SENTRY_CUDA_TRY(launch_chained(moe_combine_kernel<float>, dim3((unsigned)blocks), dim3(256), 0, st,
                (const uint4*)w.staged, m.expert_ids, m.expert_weights, d.N, vpr, d.E, d.top_k, (uint4*)m.Y));
        else if (d.dtype == SENTRY_F16)
            SENTRY_CUDA_TRY(launch_chained(moe_combine_kernel<__half>, dim3((unsigned)blocks), dim3(256), 0, st,
                (const uint4*)w.staged, m.expert_ids, m.expert_weights, d.N, vpr, d.E, d.top_k, (uint4*)m.Y));
        else
            SENTRY_CUDA_TRY(launch_chained(moe_combine_kernel<__nv_bfloat16>, dim3((unsigned)blocks), dim3(256), 0, st,
                (const uint4*)w.staged, m.expert_ids, m.expert_weights, d.N, vpr, d.E, d.top_k, (uint4*)m.Y));
    }
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}
