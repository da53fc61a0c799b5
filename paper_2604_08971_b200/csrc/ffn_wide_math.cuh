// Arithmetic of ffn_wide.cu that needs no GPU, so that a CPU test can compile it too: the GELU of GEMM 1's epilogue, and
// the tiles' widths.
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define SENTRY_HD __host__ __device__ __forceinline__
#else
#define SENTRY_HD inline
#endif

// gelu(z) = z Phi(z), to the accuracy of the library's erff form 0.5 z (1 + erff(z / sqrt 2)) or better everywhere:
//   |z| < 1   z / 2 + z^2 P(z^2), the odd part of Phi as a polynomial (own minimax fit, 7e-9 |z|)
//   else      max(z, 0) - |z| Q(|z|), Q(a) = exp(-a^2/2) R(1 / (1 + 0.32 a)) the tail of the normal distribution (own minimax fit
//             of R, 8e-9 |z|, weighted by Q down to 1e-2 so that small tails keep their digits)
// The tail form alone carries the errors of exp and reciprocal into the result at half their size near 0; here with
// Q(1) = 0.16 at most.  rcp and ex2 are the caller's 1/x and 2^x.  Error over |z| on the device against float64 (1e7 values each), here
// / erff form / tail form alone: at most 9.5e-8 / 1.2e-7 / 2.5e-7; RMS for normal z of deviation 0.03 2.6e-8 / 3.7e-8 / 1.4e-7, of 0.3
// 3.0e-8 / 4.1e-8 / 9.1e-8, of 1 2.9e-8 / 3.8e-8 / 3.7e-8, of 3 2.2e-8 / 3.1e-8 / 2.2e-8.  No sum overflows: a large finite z is
// returned.  NaN stays NaN; an infinite z gives NaN, as the second GEMM would from its stored head and remainder (inf - inf).
template <class Rcp, class Ex2>
SENTRY_HD float gelu_two_part(float z, Rcp rcp, Ex2 ex2) {
    const float a = fabsf(z), s = z * z;
    const float t = rcp(fmaf(0.32f, a, 1.f)), e = ex2(s * -0.72134752f);
    float r = fmaf(-0.0766471736f, t, 0.164664529f);
    r = fmaf(r, t, 0.0252527479f);
    r = fmaf(r, t, 0.134429036f);
    r = fmaf(r, t, 0.124188135f);
    r = fmaf(r, t, 0.127972288f);
    r = fmaf(r, t, -1.06966041e-05f);
    float p = fmaf(9.24683689e-05f, s, -0.00116535074f);
    p = fmaf(p, s, 0.0099641668f);
    p = fmaf(p, s, -0.06648873f);
    p = fmaf(p, s, 0.398942199f);
    const float near = fmaf(s, p, 0.5f * z), far = fmaf(-a, r * e, fmaxf(z, 0.f));
    return s < 1.f ? near : far;
}

// Columns of a tile of GEMM 1 (first) and 2: a multiple of 32 from 64 to wide_bn_max; wide_ctas of them run on an SM.
SENTRY_HD constexpr int wide_bn_max(bool first) { return first ? 160 : 192; }
SENTRY_HD constexpr int wide_ctas(bool first) { return first ? 2 : 1; }
// Column tiles that a launch has CTAs for: what the narrowest tiles need, since the width is chosen on the device.
SENTRY_HD constexpr int wide_grid_cols(int cols) { return (cols + 63) / 64; }
// The width where R row tiles have `cols` columns: the rounds times what a K block costs in shared-memory traffic, which is that
// of A and the columns of B (in units of B's).
SENTRY_HD int wide_bn(bool first, int R, int cols, int sm_count) {
    const int slots = sm_count * wide_ctas(first);
    int best = 64, best_cost = 0x7fffffff;
    for (int bn = 64; bn <= wide_bn_max(first); bn += 32) {
        const int items = R * ((cols + bn - 1) / bn), cost = (items + slots - 1) / slots * ((first ? 128 : 170) + bn);
        if (cost < best_cost) { best = bn; best_cost = cost; }
    }
    return best;
}
