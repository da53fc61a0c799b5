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

// Forms of the two GEMMs: the first, with two CTAs per SM; the second with one CTA per SM, which has room for four stages of up to 192
// columns; the second with two, which have two stages of 128 columns each, and one's epilogue runs beside the other's arithmetic.
enum WideForm { kWideFirst, kWideSecondOne, kWideSecondTwo };
// Columns of a tile: a multiple of 32 from 64 to wide_bn_max; wide_ctas of them run on an SM.
SENTRY_HD constexpr int wide_bn_max(int form) { return form == kWideFirst ? 160 : form == kWideSecondOne ? 192 : 128; }
SENTRY_HD constexpr int wide_ctas(int form) { return form == kWideSecondOne ? 1 : 2; }
// Column tiles that a launch has CTAs for: what the narrowest tiles need, since the width is chosen on the device.
SENTRY_HD constexpr int wide_grid_cols(int cols) { return (cols + 63) / 64; }
// The width where R row tiles have `cols` columns: the tiles an SM gets times what a K block costs in shared-memory traffic, which is
// that of A and the columns of B (in units of B's).  The two CTAs of an SM share that traffic, so they count as one: by the rounds of
// pairs instead, 44 row tiles with 1024 columns took 96 columns and 46.7 us for a call of 512 channels (128 columns: 43.2).
SENTRY_HD int wide_bn(int form, int R, int cols, int sm_count) {
    int best = 64, best_cost = 0x7fffffff;
    for (int bn = 64; bn <= wide_bn_max(form); bn += 32) {
        const int items = R * ((cols + bn - 1) / bn), cost = (items + sm_count - 1) / sm_count * ((form == kWideFirst ? 128 : 170) + bn);
        if (cost < best_cost) { best = bn; best_cost = cost; }
    }
    return best;
}
// The second GEMM's form.  A CTA alone is the faster one where an SM has a single tile, since nothing could run beside it (one / two, us
// a call on materialised weights: 3 row tiles of d_model 192, 800 channels 19.1 / 21.8; 10 of 768, 1200 27.4 / 28.5; 34 of 640, 1200
// 37.2 / 40.3; 40 of 320, 3000 67.8 / 77.5; 120 of 192, 2000 103.5 / 110.7), and loses 5 to 16 % from the second tile on (60 of 512,
// 500 34.2 / 29.7; 90 of 320, 500 39.4 / 35.2; 40 of 640, 2000 72.0 / 62.1; 300 of 1024, 200 171.7 / 138.4), or with few K blocks
// (75 of 192, 64 channels 15.4 / 14.7).  The host knows the rows of a call in which every token is present: with several lists,
// the sign of samples that miss modalities, two thirds of them and half a tile for every list.
inline bool wide_second_one(int D, int k_c, long long rows, bool token_ids, int n_lists, int most_tiles, int sm_count) {
    long long R = (rows + 127) / 128;
    if (n_lists > 1) R = (token_ids ? R * 2 / 3 : R) + n_lists / 2;
    if (R > most_tiles) R = most_tiles;
    return k_c >= 200 && R * ((D + wide_bn_max(kWideSecondOne) - 1) / wide_bn_max(kWideSecondOne)) <= sm_count;
}
