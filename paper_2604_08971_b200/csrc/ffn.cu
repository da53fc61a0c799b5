// Channel-compacted FFN (Section 4.6): y = gelu(x W1[:, N]) W2[N, :].
// This file holds the row plan, the weight gather ("materialising" W1', W2')
// and the plain-ALU fp32-accumulate kernel; the tensor-core kernels live
// in ffn_tmem.cu, ffn_tc.cu and ffn_wide.cu and share the plan.
#include <math.h>

#include "common.cuh"
#include <cuda_fp8.h>

#include "ffn_plan.cuh"

namespace {

constexpr int kGenericTileRows = 16, kGenericFewRows = 4;   // rows of a plain-ALU tile
constexpr int kGenericThreads = 256;
constexpr int kTcTileRows = 128;

// One launch prepares everything the main kernel needs.  Block ranges:
//   [0, P)              row tables of G samples each (P = ceil(B / G)): every block finds by itself where its samples'
//                       rows start (a scan over all samples' lists and present-row counts, so no separate planning
//                       launch is needed); block 0 also writes the per-list offsets and tile counts.  G = 1 for small
//                       batches, whose blocks are then all in flight at once; from kGroupPlanB samples on the scan is
//                       what a block does, and eight samples share it
//   [P, P + B*zsplit)   (not with the fused kernel, which does it itself) zero rows of Y for the absent tokens of a sample (slices of its rows)
//   [.., + prepack)     the weight gather, which "materialises" the pruned W1', W2' per list:
//     layout 0 (plain-ALU kernel): W1g [l][D][kc_pad], W2g [l][kc_pad][D]
//     layout 1 (tensor-core kernel, both K-major): W1c [l][kc_pad][D], W2c [l][D][kc_pad]
//     columns / rows n >= k_c are zero.
constexpr int kGroupPlanB = 1024;
constexpr int kPlanListsSmem = 1024;   // lists whose row counts block 0 keeps in shared memory

template <int G>
__device__ __forceinline__ void plan_block(const int32_t* __restrict__ ids, const uint32_t* __restrict__ masks,
                                           const int32_t* __restrict__ list_of_sample, int B, int Tlen, int tile_rows,
                                           const FfnPlan& p, int n_lists, unsigned int* status) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __shared__ int s_cnt[32];
    __shared__ int red[66];
    __shared__ int s_before[G][8];
    __shared__ int s_rows[kPlanListsSmem];
    const int b0 = blockIdx.x * G;
    const bool first_block = blockIdx.x == 0;
    if (threadIdx.x < 32) s_cnt[threadIdx.x] = 0;
    if (first_block)
        for (int l = threadIdx.x; l < min(n_lists, kPlanListsSmem); l += blockDim.x) s_rows[l] = 0;
    __syncthreads();
    // the first sample of this thread's share and the block's own ones, requested before the token counts are there
    const int bb_first = threadIdx.x;
    int l_first = 0, own_l[G];
    uint32_t mask_first = 0u, own_mask[G];
    if (bb_first < B) {
        if (list_of_sample != nullptr) l_first = list_of_sample[bb_first];
        if (ids != nullptr) mask_first = masks[bb_first];
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
        own_l[g] = b0 + g < B && list_of_sample != nullptr ? list_of_sample[b0 + g] : 0;
        own_mask[g] = b0 + g < B && ids != nullptr ? masks[b0 + g] : 0xffffffffu;
    }
    if (ids != nullptr) {
        // eight of a thread's tokens on the way at once (with one, 16 round trips at 4096 tokens: 15 us of this kernel, now 10)
        for (int t0 = 0; t0 < Tlen; t0 += 8 * blockDim.x) {
            int m[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int t = t0 + u * blockDim.x + threadIdx.x;
                m[u] = t < Tlen ? ids[t] : -1;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int t = t0 + u * blockDim.x + threadIdx.x;
                if (t0 + u * (int)blockDim.x >= Tlen) break;
                if (t < Tlen && (m[u] < 0 || m[u] >= 32) && first_block) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
                // tokens of a modality lie together: one shared-memory atomic per warp and modality
                const unsigned peers = __match_any_sync(0xffffffffu, m[u]);
                if (m[u] >= 0 && m[u] < 32 && lane == __ffs(peers) - 1) atomicAdd(&s_cnt[m[u]], __popc(peers));
            }
        }
        __syncthreads();
    }
    auto present_rows = [&](uint32_t mask) {
        if (ids == nullptr) return Tlen;
        int n = 0;
        while (mask) { const int m = __ffs(mask) - 1; n += s_cnt[m]; mask &= mask - 1; }
        return n;
    };
    auto checked = [&](int l) {
        if (l < 0 || l >= n_lists) {
            if (first_block) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
            l = 0;
        }
        return l;
    };
    // rows of all samples in earlier lists, and of earlier samples in the sample's list
    int my_list[G], before[G];
#pragma unroll
    for (int g = 0; g < G; ++g) { my_list[g] = b0 + g < B ? checked(own_l[g]) : -1; before[g] = 0; }
    auto count = [&](int bb, int l_raw, uint32_t mask) {
        const int l = checked(l_raw), r = present_rows(mask);
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (l < my_list[g] || (l == my_list[g] && bb < b0 + g)) before[g] += r;
        if (first_block) {
            if (r == 0) atomicOr(status, SENTRY_STATUS_BIT_EMPTY_MASK);
            if (n_lists <= kPlanListsSmem) atomicAdd(&s_rows[l], r);
        }
    };
    if (bb_first < B) count(bb_first, l_first, mask_first);
    // the rest of a large batch four samples at a time (4096 samples, one at a time: 21 us of this kernel; the step 681 -> 677)
    for (int bb = bb_first + blockDim.x; bb < B; bb += 4 * blockDim.x) {
        int l4[4];
        uint32_t m4[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int at = min(bb + u * (int)blockDim.x, B - 1);
            l4[u] = list_of_sample != nullptr ? list_of_sample[at] : 0;
            m4[u] = ids != nullptr ? masks[at] : 0u;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (bb + u * (int)blockDim.x < B) count(bb + u * blockDim.x, l4[u], m4[u]);
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
        before[g] = __reduce_add_sync(0xffffffffu, before[g]);
        if (lane == 0) s_before[g][wid] = before[g];
    }
    __syncthreads();
    if (first_block) {
        // per-list totals -> list offsets and tile counts
        if (n_lists <= kPlanListsSmem) {
            if (wid == 0) {
                int row0 = 0, tile0 = 0;
                for (int l0 = 0; l0 < n_lists; l0 += 32) {
                    const int l = l0 + lane;
                    const int r = l < n_lists ? s_rows[l] : 0, c = (r + tile_rows - 1) / tile_rows;
                    int ir = r, ic = c;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int vr = __shfl_up_sync(0xffffffffu, ir, o), vc = __shfl_up_sync(0xffffffffu, ic, o);
                        if (lane >= o) { ir += vr; ic += vc; }
                    }
                    if (l < n_lists) { p.list_row0[l] = row0 + ir - r; p.tile_start[l] = tile0 + ic - c; }
                    row0 += __shfl_sync(0xffffffffu, ir, 31);
                    tile0 += __shfl_sync(0xffffffffu, ic, 31);
                }
                if (lane == 0) { p.list_row0[n_lists] = row0; p.tile_start[n_lists] = tile0; }
            }
        } else {   // very many lists: a pass over the samples for each
            int row0 = 0, tile0 = 0;
            for (int l = 0; l < n_lists; ++l) {
                int rows = 0;
                for (int bb = threadIdx.x; bb < B; bb += blockDim.x)
                    if (checked(list_of_sample ? list_of_sample[bb] : 0) == l) rows += present_rows(ids != nullptr ? masks[bb] : 0u);
                rows = block_sum_int(rows, red);
                if (threadIdx.x == 0) { p.list_row0[l] = row0; p.tile_start[l] = tile0; }
                row0 += rows;
                tile0 += (rows + tile_rows - 1) / tile_rows;
            }
            if (threadIdx.x == 0) { p.list_row0[n_lists] = row0; p.tile_start[n_lists] = tile0; }
        }
    }
    // present tokens of the samples, ascending -> row table; eight pieces of 32 tokens at a time
    auto pieces = [&](int pc, int p1, uint32_t mask, unsigned (&bm)[8]) {
        int m[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int t = (pc + u) * 32 + lane;
            m[u] = pc + u < p1 && t < Tlen ? (ids != nullptr ? ids[t] : 0) : -1;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) bm[u] = __ballot_sync(0xffffffffu, m[u] >= 0 && m[u] < 32 && ((mask >> m[u]) & 1u));
    };
    auto put = [&](int b, int pc, const unsigned (&bm)[8], int& base) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if ((bm[u] >> lane) & 1u) p.rowidx[base + __popc(bm[u] & ((1u << lane) - 1u))] = b * Tlen + (pc + u) * 32 + lane;
            base += __popc(bm[u]);
        }
    };
    const int n_pieces = (Tlen + 31) / 32;
    if constexpr (G > 1) {   // a warp per sample
        static_assert(G <= 8, "one warp per sample of the group");
        const int b = b0 + wid;
        if (wid < G && b < B) {
            int base = 0;
            for (int w = 0; w < nw; ++w) base += s_before[wid][w];
            if (lane == 0) p.sample_row0[b] = base;
            const uint32_t mask = ids != nullptr ? masks[b] : 0xffffffffu;
            for (int pc = 0; pc < n_pieces; pc += 8) {
                unsigned bm[8];
                pieces(pc, n_pieces, mask, bm);
                put(b, pc, bm, base);
            }
        }
    } else {                 // the whole block: every warp a run of 32-token pieces, after one count of what comes before
        const int b = b0;
        int base = 0;
        for (int w = 0; w < nw; ++w) base += s_before[0][w];
        if (threadIdx.x == 0) p.sample_row0[b] = base;
        const int per = (n_pieces + nw - 1) / nw;
        const int p0 = wid * per, p1 = min(p0 + per, n_pieces);
        unsigned bm[8];
        int mine = 0;
        for (int pc = p0; pc < p1; pc += 8) {
            pieces(pc, p1, own_mask[0], bm);
#pragma unroll
            for (int u = 0; u < 8; ++u) mine += __popc(bm[u]);
        }
        if (lane == 0) red[wid] = mine;
        __syncthreads();
        for (int w = 0; w < wid; ++w) base += red[w];
        for (int pc = p0; pc < p1; pc += 8) {
            if (per > 8) pieces(pc, p1, own_mask[0], bm);   // (with one run of eight they are still there)
            put(b, pc, bm, base);
        }
    }
}

template <typename T, int G>
__global__ void __launch_bounds__(256)
ffn_prepare_kernel(const int32_t* __restrict__ ids, const uint32_t* __restrict__ masks,
                   const int32_t* __restrict__ list_of_sample, int B, int Tlen, int zsplit,
                   int tile_rows, FfnPlan p, uint8_t* __restrict__ Y,
                   const T* __restrict__ W1, const T* __restrict__ W2,
                   const int32_t* __restrict__ kept, int n_lists, int D, int F, int k_c, int kc_pad,
                   int layout, size_t w_stride, T* __restrict__ out1, T* __restrict__ out2,
                   int early, unsigned int* status) {
    // early: the next kernel is small (one that fills the GPU waits on SMs that these blocks still need)
    if (early) grid_dependents_start();
    grid_dependency_wait();
    // w_stride: elements between the weight matrices of consecutive lists (0: every list gathers
    // from the same W1, W2; D*F: list l has its own, as the experts of a Sparse-MoE block do)
    const int plan_blocks = (B + G - 1) / G;
    if ((int)blockIdx.x < plan_blocks) {
        plan_block<G>(ids, masks, list_of_sample, B, Tlen, tile_rows, p, n_lists, status);
        return;
    }
    size_t pb = (size_t)blockIdx.x - plan_blocks;
    const size_t zero_blocks = (ids != nullptr) ? (size_t)B * zsplit : 0;
    if (pb < zero_blocks) {
        // zero the rows of absent tokens, 16 bytes per store
        const int b = (int)(pb / zsplit), part = (int)(pb % zsplit);
        const uint32_t mask = masks[b];
        const int vpr = D * (int)sizeof(T) / 16;
        const int total = Tlen * vpr;
        const int per = (total + zsplit - 1) / zsplit;
        const int end = min(total, (part + 1) * per);
        uint4* Yb = reinterpret_cast<uint4*>(Y + (size_t)b * Tlen * D * sizeof(T));
        for (int i = part * per + threadIdx.x; i < end; i += blockDim.x) {
            const int m = ids[i / vpr];
            const bool present = (m >= 0 && m < 32) && ((mask >> m) & 1u);
            if (!present) Yb[i] = make_uint4(0, 0, 0, 0);
        }
        return;
    }
    pb -= zero_blocks;
    if (layout == 1) {
        // K-major copies for the tensor-core kernels, one tile of 64 channels x 64 columns per block, transposed through
        // shared memory:  W1c[l][n][e] = W1[e][N[n]],  W2c[l][e][n] = W2[N[n]][e].  A thread has all its loads in flight at once.
        if constexpr (sizeof(T) == 2) {
            // A thread turns 16-bit elements into whole 16-byte pieces in its registers; the pieces pass through shared memory
            // (swizzled, no bank conflicts) so that eight lanes write a row's 128 bytes.  Bound by latency for one list, by L2
            // beyond (26 MB of copies at d_model 768, 1229 channels, seven lists: 24 us with element-wise shared memory and 16-byte
            // stores of 32 different rows, which L2 saw as 100 MB of sectors).
            // A block has the tile of both copies, for the same channels and columns: one set of channel numbers, twice the loads on
            // the way (19.6 -> 16.5 us there).
            __shared__ __align__(16) uint4 s_piece[2][64 * 8];
            const int tiles_n = kc_pad / 64, tiles_e = D / 64;
            const size_t per_list = (size_t)tiles_n * tiles_e;
            const int l = (int)(pb / per_list);
            const int tn = (int)((pb % per_list) / tiles_e), te = (int)(pb % tiles_e);
            const int n0 = tn * 64, e0 = te * 64, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
            auto channel = [&](int n) {
                if (n >= k_c) return -1;
                const int ch = kept[(size_t)l * k_c + n];
                if (ch >= 0 && ch < F) return ch;
                if (te == 0) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
                return -1;
            };
            // W1: thread = channel tid & 63, columns 16 (tid >> 6) ..;  W2: warp = channels 8 wid .., lane = columns 2 lane, 2 lane + 1
            const int n = tid & 63, c0 = 2 * (tid >> 6);
            const int ch1 = channel(n0 + n), mine = lane < 8 ? channel(n0 + 8 * wid + lane) : -1;
            const uint16_t* src1 = reinterpret_cast<const uint16_t*>(W1 + (size_t)l * w_stride) + (size_t)(e0 + 8 * c0) * F + ch1;
            uint32_t v[16], w[8];
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = ch1 >= 0 ? src1[(size_t)i * F] : 0u;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int ch = __shfl_sync(0xffffffffu, mine, i);
                w[i] = ch >= 0 ? *reinterpret_cast<const uint32_t*>(W2 + (size_t)l * w_stride + (size_t)ch * D + e0 + 2 * lane) : 0u;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h)
                s_piece[0][n * 8 + ((c0 + h) ^ (n & 7))] = make_uint4(v[8 * h] | v[8 * h + 1] << 16, v[8 * h + 2] | v[8 * h + 3] << 16,
                                                                      v[8 * h + 4] | v[8 * h + 5] << 16, v[8 * h + 6] | v[8 * h + 7] << 16);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t sel = h == 0 ? 0x5410u : 0x7632u;
                s_piece[1][(2 * lane + h) * 8 + (wid ^ (lane & 7))] =
                    make_uint4(__byte_perm(w[0], w[1], sel), __byte_perm(w[2], w[3], sel), __byte_perm(w[4], w[5], sel),
                               __byte_perm(w[6], w[7], sel));
            }
            __syncthreads();
            T* dst1 = out1 + ((size_t)l * kc_pad + n0) * D + e0;
            T* dst2 = out2 + ((size_t)l * D + e0) * kc_pad + n0;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int r = (tid >> 3) + 32 * j, c = tid & 7;
                *reinterpret_cast<uint4*>(dst1 + (size_t)r * D + c * 8) = s_piece[0][r * 8 + (c ^ (r & 7))];
                *reinterpret_cast<uint4*>(dst2 + (size_t)r * kc_pad + c * 8) = s_piece[1][r * 8 + (c ^ ((r >> 1) & 7))];
            }
        }
        if constexpr (sizeof(T) == 1) {   // element by element
            constexpr int VEC = 16;           // elements of a 16-byte piece
            constexpr int PITCH = 64 + 4;     // elements; odd number of words
            __shared__ __align__(16) T s_tile[64 * PITCH];
            __shared__ int s_ch[64];
            const int tiles_n = kc_pad / 64, tiles_e = D / 64;
            const size_t per_list = (size_t)tiles_n * tiles_e;
            const int which = (int)(pb / (per_list * n_lists));
            pb -= (size_t)which * per_list * n_lists;
            const int l = (int)(pb / per_list);
            const int tn = (int)((pb % per_list) / tiles_e), te = (int)(pb % tiles_e);
            const int n0 = tn * 64, e0 = te * 64;
            const T* W1l = W1 + (size_t)l * w_stride;
            const T* W2l = W2 + (size_t)l * w_stride;
            if (threadIdx.x < 64) {
                const int n = n0 + threadIdx.x;
                int ch = -1;
                if (n < k_c) {
                    ch = kept[(size_t)l * k_c + n];
                    if (ch < 0 || ch >= F) {
                        if (which == 0 && te == 0) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
                        ch = -1;
                    }
                }
                s_ch[threadIdx.x] = ch;
            }
            __syncthreads();
            const T zero = from_f32<T>(0.f);
            T* dst;
            size_t ld;
            if (which == 0) {
                // s_tile[e][n]
                const int tx = threadIdx.x & 31, wy = threadIdx.x >> 5;   // 8 warps
                const int c0 = s_ch[tx], c1 = s_ch[tx + 32];
                T v0[8], v1[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const T* row = W1l + (size_t)(e0 + wy + 8 * i) * F;
                    v0[i] = c0 >= 0 ? row[c0] : zero;
                    v1[i] = c1 >= 0 ? row[c1] : zero;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    s_tile[(wy + 8 * i) * PITCH + tx] = v0[i];
                    s_tile[(wy + 8 * i) * PITCH + tx + 32] = v1[i];
                }
                dst = out1 + ((size_t)l * kc_pad + n0) * D + e0;
                ld = D;
            } else {
                // s_tile[n][e]
                for (int i = threadIdx.x; i < 64 * 64 / VEC; i += 256) {
                    const int nn = i / (64 / VEC), c = i % (64 / VEC);
                    const int ch = s_ch[nn];
                    uint4 v = make_uint4(0, 0, 0, 0);
                    if (ch >= 0) {
                        const T* src = W2l + (size_t)ch * D + e0 + c * VEC;
                        v = *reinterpret_cast<const uint4*>(src);
                    }
                    const T* p8 = reinterpret_cast<const T*>(&v);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) s_tile[nn * PITCH + c * VEC + e] = p8[e];
                }
                dst = out2 + ((size_t)l * D + e0) * kc_pad + n0;
                ld = kc_pad;
            }
            __syncthreads();
            // column r of s_tile -> row r of the copy
            for (int i = threadIdx.x; i < 64 * 64 / VEC; i += 256) {
                const int r = i % 64, c = i / 64;
                uint4 v;
                T* p8 = reinterpret_cast<T*>(&v);
#pragma unroll
                for (int e = 0; e < VEC; ++e) p8[e] = s_tile[(c * VEC + e) * PITCH + r];
                *reinterpret_cast<uint4*>(dst + (size_t)r * ld + c * VEC) = v;
            }
            return;
        }
        return;
    }
    const size_t per = (size_t)kc_pad * D;
    const size_t blocks_per = (per + 255) / 256;
    const int which = (int)(pb / (blocks_per * n_lists));
    pb -= (size_t)which * blocks_per * n_lists;
    const int l = (int)(pb / blocks_per);
    const size_t i = (pb % blocks_per) * 256 + threadIdx.x;
    if (i >= per) return;
    const int32_t* N = kept + (size_t)l * k_c;
    if (which == 0) {
        // W1: destination-major index so that writes coalesce
        const int e = (int)(i / kc_pad), n = (int)(i % kc_pad);
        T v = from_f32<T>(0.f);
        if (n < k_c) {
            const int ch = N[n];
            if (ch >= 0 && ch < F) v = W1[(size_t)l * w_stride + (size_t)e * F + ch];
            else if (e == 0) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
        }
        out1[(size_t)l * per + i] = v;
    } else {
        const int n = (int)(i / D), e = (int)(i % D);
        T v = from_f32<T>(0.f);
        if (n < k_c) {
            const int ch = N[n];
            if (ch >= 0 && ch < F) v = W2[(size_t)l * w_stride + (size_t)ch * D + e];
        }
        out2[(size_t)l * per + i] = v;
    }
}

// The weight gather from FP8 storage: W1q [D,F] and W2q [F,D] hold e4m3 codes (4 exponent bits, 3
// fraction bits, bias 7, no infinities), each with one fp32 scale; element = decode(code) * scale,
// rounded once to the compute type T.  Same destination layouts as the gather above; a one-off
// (materialise-once) step, so one thread per destination element is enough.
template <typename T>
__global__ void __launch_bounds__(256)
ffn_prepack_fp8_kernel(const uint8_t* __restrict__ W1q, const uint8_t* __restrict__ W2q, float s1, float s2,
                       const int32_t* __restrict__ kept, int n_lists, int D, int F, int k_c, int kc_pad,
                       int layout, T* __restrict__ out1, T* __restrict__ out2, unsigned int* status) {
    const size_t per = (size_t)kc_pad * D;
    const size_t blocks_per = (per + 255) / 256;
    size_t pb = blockIdx.x;
    const int which = (int)(pb / (blocks_per * n_lists));
    pb -= (size_t)which * blocks_per * n_lists;
    const int l = (int)(pb / blocks_per);
    const size_t i = (pb % blocks_per) * 256 + threadIdx.x;
    if (i >= per) return;
    const int32_t* N = kept + (size_t)l * k_c;
    auto decode = [](uint8_t code) {
        __nv_fp8_e4m3 q;
        q.__x = code;
        return float(q);
    };
    int n, e;
    if (which == 0) {
        if (layout == 0) { e = (int)(i / kc_pad); n = (int)(i % kc_pad); }
        else             { n = (int)(i / D);      e = (int)(i % D); }
    } else {
        if (layout == 0) { n = (int)(i / D);      e = (int)(i % D); }
        else             { e = (int)(i / kc_pad); n = (int)(i % kc_pad); }
    }
    T v = from_f32<T>(0.f);
    if (n < k_c) {
        const int ch = N[n];
        if (ch >= 0 && ch < F)
            v = which == 0 ? from_f32<T>(decode(W1q[(size_t)e * F + ch]) * s1) : from_f32<T>(decode(W2q[(size_t)ch * D + e]) * s2);
        else if (which == 0 && e == 0) atomicOr(status, SENTRY_STATUS_BIT_BAD_INDEX);
    }
    (which == 0 ? out1 : out2)[(size_t)l * per + i] = v;
}

__device__ __forceinline__ float gelu_erf(float z) {
    return 0.5f * z * (1.0f + erff(z * 0.70710678118654752440f));
}

// Plain-ALU fused pair on a tile of R present rows.  grid = tile upper bound.  SLOTS: 256-column pieces of d_model that
// fit D.  A thread owns a hidden channel, then an output column, of all R rows: R multiply-adds per weight it loads.  On
// a few rows that is a chain of weight loads from L2, so three groups of 8 are on the way while a fourth is used, and the rows'
// side comes from shared memory four values at a time.  64 fp32 rows of d_model 64, 128 channels: the call 28 -> 11 us.
template <typename T, int SLOTS, int R>
__global__ void __launch_bounds__(kGenericThreads)
ffn_generic_kernel(const T* __restrict__ X, const T* __restrict__ W1g, const T* __restrict__ W2g,
                   FfnPlan plan, int n_lists, int Tlen, int D, int k_c, int kc_pad,
                   T* __restrict__ Y) {
    constexpr int KB = 8, NB = 4;
    extern __shared__ __align__(16) float s_f[];
    float* s_x = s_f;                   // [R][D]
    float* s_h = s_f + (size_t)R * D;   // [R][256]
    __shared__ long long s_row[R], s_out[R];
    grid_dependents_start_if_small();
    grid_dependency_wait();
    int l, row0, n_rows;
    if (!ffn_tile_lookup(plan, n_lists, blockIdx.x, R, l, row0, n_rows)) return;
    if (threadIdx.x < R) {
        s_row[threadIdx.x] = threadIdx.x < n_rows ? (long long)plan.rowidx[row0 + threadIdx.x] : -1;
        s_out[threadIdx.x] = threadIdx.x < n_rows
                                 ? (long long)(plan.rowout ? plan.rowout : plan.rowidx)[row0 + threadIdx.x] : -1;
    }
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < R * D; i += kGenericThreads) {
        const int r = i / D, e = i % D;
        s_x[i] = s_row[r] >= 0 ? to_f32<T>(X[(size_t)s_row[r] * D + e]) : 0.f;
    }
    const T* w1 = W1g + (size_t)l * D * kc_pad;
    const T* w2 = W2g + (size_t)l * kc_pad * D;
    // acc[r] += sum over k of row[r][k] * col[k * stride], k ascending; n is a multiple of 8
    auto dot_rows = [](float (&acc)[R], const float* row, int row_stride, const T* col, size_t stride, int n) {
        float w[NB][KB];
#pragma unroll
        for (int i = 0; i < NB - 1; ++i)
            if (i * KB < n)
#pragma unroll
                for (int j = 0; j < KB; ++j) w[i][j] = to_f32<T>(col[(size_t)(i * KB + j) * stride]);
#pragma unroll 1
        for (int k0 = 0; k0 < n; k0 += NB * KB) {
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const int k = k0 + i * KB, ahead = k + (NB - 1) * KB;
                if (k >= n) break;
                if (ahead < n)
#pragma unroll
                    for (int j = 0; j < KB; ++j) w[(i + NB - 1) % NB][j] = to_f32<T>(col[(size_t)(ahead + j) * stride]);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float4* x = reinterpret_cast<const float4*>(row + r * row_stride + k);
#pragma unroll
                    for (int q = 0; q < KB / 4; ++q) {
                        const float4 v = x[q];
                        acc[r] = fmaf(v.x, w[i][4 * q], acc[r]);
                        acc[r] = fmaf(v.y, w[i][4 * q + 1], acc[r]);
                        acc[r] = fmaf(v.z, w[i][4 * q + 2], acc[r]);
                        acc[r] = fmaf(v.w, w[i][4 * q + 3], acc[r]);
                    }
                }
            }
        }
    };
    float y[SLOTS][R];
#pragma unroll
    for (int s = 0; s < SLOTS; ++s)
#pragma unroll
        for (int r = 0; r < R; ++r) y[s][r] = 0.f;
    __syncthreads();
    for (int c0 = 0; c0 < k_c; c0 += kGenericThreads) {
        const int n = c0 + threadIdx.x;
        float hacc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) hacc[r] = 0.f;
        if (n < k_c) dot_rows(hacc, s_x, D, w1 + n, kc_pad, D);
#pragma unroll
        for (int r = 0; r < R; ++r)
            s_h[r * kGenericThreads + threadIdx.x] = (n < k_c) ? gelu_erf(hacc[r]) : 0.f;
        __syncthreads();
        const int cn = min(kGenericThreads, kc_pad - c0);   // (channels past k_c: zero weights, zero hidden values)
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) {
            const int e = s * kGenericThreads + threadIdx.x;
            if (e < D) dot_rows(y[s], s_h, kGenericThreads, w2 + (size_t)c0 * D + e, D, cn);
        }
        __syncthreads();
    }
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
        const int e = s * kGenericThreads + threadIdx.x;
        if (e < D) {
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (s_out[r] >= 0) Y[(size_t)s_out[r] * D + e] = from_f32<T>(y[s][r]);
        }
    }
}

// Weights as K-major chunk-padded copies (either tensor-core form), tiles of 128 rows.
bool k_major(const sentry_ffn_desc& d) { return ffn_tc_supported(d) || ffn_wide_supported(d); }
int tile_rows_for(const sentry_ffn_desc& d) {
    if (k_major(d)) return kTcTileRows;
    // tiles of 4 while they leave an SM to each: shorter chains, and the weights they read more often come from L2
    return (long long)d.B * d.T <= kGenericFewRows * kSmCount ? kGenericFewRows : kGenericTileRows;
}

template <typename T>
int launch_generic(const FfnArgs& a, const FfnPlan& plan, const void* w1p, const void* w2p, int kc_pad, int max_tiles,
                   cudaStream_t st) {
    const sentry_ffn_desc& d = a.d;
    const int rows = tile_rows_for(d);
    const size_t smem = ((size_t)rows * d.D + (size_t)rows * kGenericThreads) * 4;
    const bool few = rows == kGenericFewRows, one = d.D <= kGenericThreads;
    auto kern = few ? (one ? ffn_generic_kernel<T, 1, kGenericFewRows> : ffn_generic_kernel<T, 4, kGenericFewRows>)
                    : (one ? ffn_generic_kernel<T, 1, kGenericTileRows> : ffn_generic_kernel<T, 4, kGenericTileRows>);
    if (smem > 40 * 1024)   // (beside the static arrays)
        SENTRY_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    SENTRY_CUDA_TRY(launch_chained(kern, dim3(max_tiles), dim3(kGenericThreads), smem, st, (const T*)a.X, (const T*)w1p,
                                   (const T*)w2p, plan, d.n_lists, d.T, d.D, d.k_c, kc_pad, (T*)a.Y));
    return SENTRY_OK;
}

struct FfnWs {
    FfnPlan plan;
    void *w1p, *w2p;
    bool ok;
    size_t used;
};

// One of W1', W2' (all lists), rounded so that the second starts 256-byte aligned.
size_t packed_half_bytes(const sentry_ffn_desc& d, int kc_pad) {
    const size_t esz = d.dtype == SENTRY_F32 ? 4 : (d.dtype == SENTRY_FP8_E4M3 ? 1 : 2);
    return align_up((size_t)d.n_lists * kc_pad * d.D * esz, 256);
}

// Row plan (and, unless the caller brings materialised weights, W1' and W2') from the workspace.
FfnWs carve(const sentry_ffn_desc& d, int kc_pad, void* ws, size_t bytes, bool with_weights) {
    WsAlloc a(ws, bytes);
    FfnWs w;
    w.plan.sample_row0 = a.take<int32_t>(d.B);
    w.plan.list_row0 = a.take<int32_t>(d.n_lists + 1);
    w.plan.tile_start = a.take<int32_t>(d.n_lists + 1);
    w.plan.rowidx = a.take<int32_t>((size_t)d.B * d.T);
    w.plan.rowout = nullptr;
    w.plan.zero_ids = nullptr;
    w.plan.zero_masks = nullptr;
    w.plan.n_rows = 0;
    w.plan.Tlen = d.T;
    w.w1p = w.w2p = nullptr;
    if (with_weights) {
        w.w1p = a.take<uint8_t>(packed_half_bytes(d, kc_pad));
        w.w2p = a.take<uint8_t>(packed_half_bytes(d, kc_pad));
    }
    w.ok = a.ok;
    w.used = a.off;
    return w;
}

// Blocks of the K-major gather: a 64 x 64 tile of both copies each (8-bit: of one).
size_t k_major_blocks(const sentry_ffn_desc& d, int kc_pad) {
    return (d.dtype == SENTRY_FP8_E4M3 ? 2 : 1) * (size_t)d.n_lists * (kc_pad / 64) * (d.D / 64);
}

int kc_pad_for(const sentry_ffn_desc& d) {
    if (ffn_tc_supported(d)) return ffn_tc_kc_pad(d.D, d.k_c);
    if (ffn_wide_supported(d)) return ffn_wide_kc_pad(d.k_c);
    return (d.k_c + 7) / 8 * 8;
}

long long tiles_bound(const sentry_ffn_desc& d) {
    const int tile_rows = tile_rows_for(d);
    return ((long long)d.B * d.T + tile_rows - 1) / tile_rows + d.n_lists;
}

}  // namespace

size_t ffn_workspace_bytes(const sentry_ffn_desc& d) {
    return carve(d, kc_pad_for(d), nullptr, 0, true).used + ffn_hidden_bytes(d, tiles_bound(d)) + 512;
}

// Scratch for the hidden activations where they leave the SM.
size_t ffn_hidden_bytes(const sentry_ffn_desc& d, long long max_tiles) {
    return ffn_wide_supported(d) ? ffn_wide_hidden_bytes(kc_pad_for(d), max_tiles) : 0;
}

size_t ffn_packed_bytes(const sentry_ffn_desc& d) { return 2 * packed_half_bytes(d, kc_pad_for(d)); }

// The weight gather alone: W1' = W1[:, N], W2' = W2[N, :] for every list into `packed`.
// (The gather moves elements and writes zeros, no arithmetic: fp16 data goes through the 16-bit
// instantiation unchanged.)
int launch_ffn_prepack(sentry_ctx* ctx, const FfnArgs& a, void* packed, cudaStream_t st) {
    const sentry_ffn_desc& d = a.d;
    const bool tc = k_major(d);
    const int kc_pad = kc_pad_for(d);
    const size_t per = (size_t)kc_pad * d.D;
    const size_t pack_blocks = tc ? k_major_blocks(d, kc_pad) : 2 * (size_t)d.n_lists * ((per + 255) / 256);
    uint8_t* w1p = (uint8_t*)packed;
    uint8_t* w2p = w1p + packed_half_bytes(d, kc_pad);
    FfnPlan none = {};
    none.rowout = nullptr;
    LaunchScope ls(ctx, KS_FFN_PREPARE, st);
    // no row-table and no zero-fill blocks (B = 0, no ids): every block gathers weights
    if (d.dtype == SENTRY_FP8_E4M3) {
        if (!tc) return SENTRY_ERR_UNSUPPORTED;
        SENTRY_CUDA_TRY(launch_chained(ffn_prepare_kernel<uint8_t, 1>, dim3((unsigned)pack_blocks), dim3(256), 0, st,
            nullptr, nullptr, nullptr, 0, d.T, 1, kTcTileRows, none, nullptr, (const uint8_t*)a.W1, (const uint8_t*)a.W2,
            a.kept, d.n_lists, d.D, d.F, d.k_c, kc_pad, 1, a.w_stride, w1p, w2p, 0, a.status));
    } else if (d.dtype == SENTRY_F32)
        SENTRY_CUDA_TRY(launch_chained(ffn_prepare_kernel<float, 1>, dim3((unsigned)pack_blocks), dim3(256), 0, st,
            nullptr, nullptr, nullptr, 0, d.T, 1, kGenericTileRows, none, nullptr, (const float*)a.W1,
            (const float*)a.W2, a.kept, d.n_lists, d.D, d.F, d.k_c, kc_pad, 0, a.w_stride, (float*)w1p, (float*)w2p, 0, a.status));
    else
        SENTRY_CUDA_TRY(launch_chained(ffn_prepare_kernel<__nv_bfloat16, 1>, dim3((unsigned)pack_blocks), dim3(256), 0, st,
            nullptr, nullptr, nullptr, 0, d.T, 1, tc ? kTcTileRows : kGenericTileRows, none, nullptr,
            (const __nv_bfloat16*)a.W1, (const __nv_bfloat16*)a.W2, a.kept, d.n_lists, d.D, d.F, d.k_c, kc_pad,
            tc ? 1 : 0, a.w_stride, (__nv_bfloat16*)w1p, (__nv_bfloat16*)w2p, 0, a.status));
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}

int launch_ffn_prepack_fp8(sentry_ctx* ctx, const sentry_ffn_desc& d, const uint8_t* W1q, const uint8_t* W2q, float s1,
                           float s2, const int32_t* kept, void* packed, cudaStream_t st) {
    const bool tc = k_major(d);
    const int kc_pad = kc_pad_for(d);
    const size_t per = (size_t)kc_pad * d.D;
    const unsigned grid = (unsigned)(2 * (size_t)d.n_lists * ((per + 255) / 256));
    uint8_t* w1p = (uint8_t*)packed;
    uint8_t* w2p = w1p + packed_half_bytes(d, kc_pad);
    const int layout = tc ? 1 : 0;
    LaunchScope ls(ctx, KS_FFN_PREPARE, st);
    if (d.dtype == SENTRY_F32)
        ffn_prepack_fp8_kernel<float><<<grid, 256, 0, st>>>(W1q, W2q, s1, s2, kept, d.n_lists, d.D, d.F, d.k_c, kc_pad,
                                                           layout, (float*)w1p, (float*)w2p, ctx->d_status);
    else if (d.dtype == SENTRY_F16)
        ffn_prepack_fp8_kernel<__half><<<grid, 256, 0, st>>>(W1q, W2q, s1, s2, kept, d.n_lists, d.D, d.F, d.k_c, kc_pad,
                                                            layout, (__half*)w1p, (__half*)w2p, ctx->d_status);
    else
        ffn_prepack_fp8_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(W1q, W2q, s1, s2, kept, d.n_lists, d.D, d.F, d.k_c,
                                                                   kc_pad, layout, (__nv_bfloat16*)w1p,
                                                                   (__nv_bfloat16*)w2p, ctx->d_status);
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}

int ffn_kc_pad(const sentry_ffn_desc& d) { return kc_pad_for(d); }
int ffn_tile_rows(const sentry_ffn_desc& d) { return tile_rows_for(d); }

// The fused pair alone, on a row plan and materialised weights that are already in place.
int launch_ffn_main(sentry_ctx* ctx, const FfnArgs& a, const FfnPlan& plan, void* w1p, void* w2p, int kc_pad,
                    int max_tiles, void* hidden, cudaStream_t st) {
    const sentry_ffn_desc& d = a.d;
    if (ffn_wide_supported(d)) {
        int rc = launch_ffn_wide(ctx, a, plan, w1p, w2p, kc_pad, max_tiles, hidden, st);
        if (rc != SENTRY_OK) return rc;
    } else if (ffn_tc_supported(d)) {
        int rc = launch_ffn_tc(ctx, a, plan, w1p, w2p, kc_pad, max_tiles, st);
        if (rc != SENTRY_OK) return rc;
    } else {
        LaunchScope ls(ctx, KS_FFN_MAIN, st);
        const int rc = d.dtype == SENTRY_F32   ? launch_generic<float>(a, plan, w1p, w2p, kc_pad, max_tiles, st)
                       : d.dtype == SENTRY_F16 ? launch_generic<__half>(a, plan, w1p, w2p, kc_pad, max_tiles, st)
                                               : launch_generic<__nv_bfloat16>(a, plan, w1p, w2p, kc_pad, max_tiles, st);
        if (rc != SENTRY_OK) return rc;
    }
    SENTRY_CUDA_TRY(cudaGetLastError());
    return SENTRY_OK;
}

// packed == nullptr: gather the weights into the workspace first (every call); otherwise use the
// caller's materialised W1', W2' (launch_ffn_prepack) and only build the row plan.
int launch_ffn(sentry_ctx* ctx, const FfnArgs& a, void* ws, size_t ws_bytes, const void* packed, cudaStream_t st) {
    const sentry_ffn_desc& d = a.d;
    const bool fused = ffn_tc_supported(d), tc = k_major(d);   // tc: K-major weights, 128-row tiles
    const int kc_pad = kc_pad_for(d);
    if (d.dtype == SENTRY_FP8_E4M3 && (packed == nullptr || !fused)) return SENTRY_ERR_UNSUPPORTED;   // FP8: prepacked weights only
    FfnWs w = carve(d, kc_pad, ws, ws_bytes, packed == nullptr);
    const size_t h_at = align_up(w.used, 256), h_bytes = ffn_hidden_bytes(d, tiles_bound(d));
    if (!w.ok || h_at + h_bytes > ws_bytes) return SENTRY_ERR_WORKSPACE;
    void* hidden = (uint8_t*)ws + h_at;
    if (packed != nullptr) {
        w.w1p = const_cast<void*>(packed);
        w.w2p = (uint8_t*)w.w1p + packed_half_bytes(d, kc_pad);
    }
    const int tile_rows = tile_rows_for(d);
    if (fused && a.ids != nullptr) {   // the fused kernel writes the zero rows
        w.plan.zero_ids = a.ids;
        w.plan.zero_masks = a.masks;
        w.plan.n_rows = d.B * d.T;
    }

    {
        const size_t per = (size_t)kc_pad * d.D;
        // other kernels: enough zero-fill blocks to cover the GPU a few times over when the batch is small
        int zsplit = fused ? 0 : (4 * ctx->sm_count + d.B - 1) / d.B;
        if (!fused && zsplit < 1) zsplit = 1;
        if (zsplit > 32) zsplit = 32;
        const size_t pack_blocks = packed != nullptr ? 0
                                   : (tc ? k_major_blocks(d, kc_pad) : 2 * (size_t)d.n_lists * ((per + 255) / 256));
        // the next kernel starts early where the CTAs of its launch leave half of the SMs free: one window of 64 tokens 31.7 -> 31.3
        // us a step; on 64 windows x 1024 tokens, whose FFN has a CTA for every SM, 116 -> 119.  The wide form, whose launch has a
        // CTA for every 64 channels, a call early / not: 32 CTAs (46 rows of d_model 768, 967 channels) 23.4 / 23.8 us, 40
        // 25.3 / 25.4, 60 22.1 / 22.1, 84 24.2 / 24.0, 96 21.6 / 21.8, 100 26.3 / 26.1, 132 27.9 / 27.4, 180 29.6 / 29.6; at d_model
        // 192 not early is faster on few, too (12 CTAs 14.0 / 13.4)
        const long long next = ffn_wide_supported(d) ? ffn_wide_first_ctas(d.k_c, tiles_bound(d)) : tiles_bound(d);
        const int early = next <= ctx->sm_count / 2;
        const bool grouped = d.B >= kGroupPlanB;
        const size_t plan_blocks = grouped ? ((size_t)d.B + 7) / 8 : (size_t)d.B;
        const size_t grid = plan_blocks + (a.ids != nullptr ? (size_t)d.B * zsplit : 0) + pack_blocks;
        LaunchScope ls(ctx, KS_FFN_PREPARE, st);
#define PREPARE(TT, G) launch_chained(ffn_prepare_kernel<TT, G>, dim3((unsigned)grid), dim3(256), 0, st,                 \
            a.ids, a.masks, a.list_of_sample, d.B, d.T, zsplit, tile_rows, w.plan, (uint8_t*)a.Y, (const TT*)a.W1,    \
            (const TT*)a.W2, a.kept, d.n_lists, d.D, d.F, d.k_c, kc_pad, tc ? 1 : 0, a.w_stride, (TT*)w.w1p, (TT*)w.w2p, early, a.status)
        if (d.dtype == SENTRY_F32) { if (grouped) SENTRY_CUDA_TRY(PREPARE(float, 8)); else SENTRY_CUDA_TRY(PREPARE(float, 1)); }
        else { if (grouped) SENTRY_CUDA_TRY(PREPARE(__nv_bfloat16, 8)); else SENTRY_CUDA_TRY(PREPARE(__nv_bfloat16, 1)); }
#undef PREPARE
    }
    SENTRY_CUDA_TRY(cudaGetLastError());
    const int max_tiles = (int)tiles_bound(d);
    return launch_ffn_main(ctx, a, w.plan, w.w1p, w.w2p, kc_pad, max_tiles, hidden, st);
}
