// Which calls of the FFN at d_model 256 (ffn_tmem.cu) pairs of CTAs take.  Host code without CUDA in it, so that a CPU test can
// compile it and hold the GPU tests' shapes to the form that they are meant for.
#pragma once

// Pairs save about a fifth of a chunk's time and cost 1.2 us once, so they pay from a number of rounds of tiles times chunks
// on: 9.  Measured with every token present, single CTAs / pairs in us: 2 chunks, 3.0 rounds 25.5 / 25.4, 5.3 rounds 35.6 / 35.0,
// 9.5 56.8 / 53.8; 3 chunks, 2.1 rounds 28.7 / 28.8, 3.5 31.4 / 30.4; 4 chunks, 2.1 rounds 33.0 / 32.7, 3.5 37.1 / 35.3; 8 chunks,
// 2.1 rounds 60.2 / 55.7.  A single chunk gains nothing at any number (3.0 rounds 18.4 / 19.5, 26 103.3 / 103.3).
// With masks max_tiles is what there is when every token is present, and a list with an odd number of tiles leaves half of
// a pair idle.  Several lists are the sign of samples that miss modalities: 18, so that half of the tokens still pay.  What
// pairs change where 100, 80, 60 and 45 % of the tokens are present, in %:
//   7 lists   512 channels  3.5 rounds  -1.3 +0.9 +3.2 +3.8    4.8  -5.2 -2.2 +1.0 +3.4    6.1  -7.9 -8.1 -4.8  0.0
//             256           6.1         -1.2  0.0 +1.6 +1.0    9.5  -5.1 -5.7 -0.2  0.0
//   1 list    512           3.0         -3.8 -2.3 +2.1 +2.6    3.5  -3.6 -1.7 -0.2 +1.4    4.1  -5.8 -3.4 -0.2 +2.9
//             256           4.1         -2.0 -0.3 +3.4 +2.5    6.1  -2.9 -1.5 +0.3 +0.2
// so 13 with one list.  Every thread adds up the lists: at most 64.
inline bool ffn_takes_pairs(bool token_ids, int n_lists, int k_c, long long max_tiles, int sm_count) {
    const int chunks = (k_c + 127) / 128, need = !token_ids ? 9 : n_lists == 1 ? 13 : 18;
    return chunks > 1 && max_tiles * chunks >= (long long)need * sm_count && n_lists <= 64;
}
