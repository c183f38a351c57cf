// routes.h -- which kernel a call of several takes, by its sizes: plain host
// functions, so that the rules can be compared with measured times anywhere.
#pragma once

#include <stddef.h>

namespace mnmt {

// what a linear of a session does (it decides the kernel with the sizes)
enum LinRole {
    LIN_LAYER,   // QKV of the encoder, FFN
    LIN_SQUARE,  // d x d: attention outputs, cross-attention queries
    LIN_CACHE,   // writes keys / values into a cache (QKV of the decoder, cross K / V)
    LIN_OUT      // vocabulary projection
};

// Does a session's linear of M >= 17 rows (n outputs, depth k, in a model of
// width d and FFN width F) run on the tcgen05 kernel, or on the kernels that read
// int8 codes?  The lines lie where whole encodes and decode steps cross (us,
// int8 / tcgen05): kernels of the two families differ in shared memory, and a
// layer that mixes them is slower than either (46 tokens, d = 512, F = 2048, per
// encode: 349 all int8, 265 all tcgen05, 308 to 318 with one linear of a layer
// changed over).
//   Layers, F <= 1024: int8 while the layer has at most 2e9 products (d 128: 4e9;
//   12800 rows of F 512 166 / 189)
//     12 layers, d 256, F 1024: 80 rows 366 / 403, 1600 rows 537 / 620, 2560 rows 684 / 691
//     12 layers, d 384, F 768: 1600 rows 574 / 678, 2560 rows 773 / 701
//     6 layers, d 512, F 1024: 1000 rows 314 / 330, 1600 rows 434 / 370
//   F > 1024 (the int8 kernel does not split a long K): tcgen05
//     6 layers, d 512, F 2048: 18 rows 302 / 255, 520 rows 376 / 355, 2560 rows 767 / 575
//     but up to 64 rows of a narrow model the int8 kernels' chunks of 16 rows:
//     6 layers, d 384, F 1536: 46 rows 189 / 238, 80 rows 259 / 245
//   Squares of such tcgen05 layers: int8 up to K = 384, and to K = 512 for up to 3e8 products
//     5120 rows, d 256: 919 / 967; 12800 rows, d 384: 1842 / 1901; d 512: 640 rows 357 / 367,
//     5120 rows 825 / 777; steps of 6 layers, 128 rows, d 512: 363 / 374
//   Cache writers: tcgen05, whose epilogue writes 16 bytes at a time (steps of 4
//     layers, d 256: 128 rows 212 / 187), but for the smallest
//   Vocabulary: 16 thousand columns and more tcgen05 (17 rows, 32000 x 512: 6.6 us
//     less), but fp32 rows of K <= 256, 65 to 128 of them (112: 1.6 less on int8);
//     fewer columns: int8 up to 6e8 products (8000 x 384: 192 rows 2.0 less, 300 rows 4.4 more)
inline bool route_linear_tc(LinRole role, int M, int d, int F, int n, int k, bool f32_out) {
    if (role == LIN_OUT) {
        if (n >= 16384) return !(f32_out && k <= 256 && M > 64 && M <= 128);
        return (double)M * n * k > 6e8;
    }
    if (role == LIN_CACHE) return !(d <= 128 && M <= 64);
    if (M <= 64 && d < 512) return false;
    if (F <= 1024 && d <= 512 && (double)M * (4.0 * d * d + 2.0 * d * F) <= (d <= 128 ? 4e9 : 2e9)) return false;
    return role != LIN_SQUARE || d > 512 || (d > 384 && (double)M * n * k > 3e8);
}

// Output tiles of a tcgen05 linear: 256 x 256 or 256 x 128 on CTA pairs, 128 x 256,
// 128 x 128 or (split K where it leaves SMs idle) 128 x 64 on single CTAs.
enum TcTiles { TC_PAIR256, TC_PAIR128, TC_WIDE, TC_128, TC_NARROW };

// sms SMs, `pairs` CTA pairs resident at once; nkb k-blocks of 64; f32: fp32
// outputs; rows16: output rows that 16-byte stores can write.
//   Codes and argmax: a pair starts later (cluster, 512 TMEM columns) and its tile
//   takes longer, and K above 1024 leaves 256 columns one accumulator buffer, so by
//   time, t + a nkb + waves x (b + c nkb) us, fitted to 2300 calls of 300 to 16384
//   rows (K 64 to 2048; 2 to 4 % rms, with two chunks 3 to 8 %), with 3 % asked for
//   before leaving 128 x 128, or up to K = 512 pairs for wide (6400 x 1536, K = 512
//   pair256 15.3, wide 15.1 alone, but 1383 / 1392 a first step).
//   Measured (128 x 128 / wide / pair256): 4000 x 2048, K = 64 13.7 / 11.6 / 12.7, K = 512 18.0
//   / 14.2 / 15.9; 3000 x 2048, K = 1024 20.6 / 17.9 / 18.7, K = 2048 33.3 / 29.9 / 29.6; 1500 x
//   2048, K = 512 10.6 / 9.5 / 11.6
//   Rows that cannot be stored 16 bytes at a time go through the pairs' staging
//   blocks (3000 x 1000, K = 512: 51.7 / 58.2 / 25.1).
//   fp32 outputs of 128 x 128 tiles are slower: one wave of pairs against two of
//   those (M 5000, N 512, residual 14.7 / 20.2; M 300, N 8192 12.8 / 14.6); with
//   equal waves they are not.
//   pair128: one wave where 128 x 64 tiles need two and K is long (M 4000, N 512,
//   residual: K 2048 18.1 / 23.1, K 1024 13.9 / 15.1, K 512 equal; M 2300, N 1024,
//   K 1024, codes 11.9 / 13.8).
//   fp32 wide: one wave that would be two of 128 x 128 (M 2400, N 2048, K 512, residual
//   20.1 / 21.1).
inline TcTiles route_tc_tiles(int M, int N, int nkb, bool f32, bool argmax, bool rows16, int sms, int pairs) {
    const auto up = [](long a, long b) { return (a + b - 1) / b; };
    const long mt = up(M, 128), mt2 = up(M, 256);
    const long t128 = mt * up(N, 128), wide = mt * up(N, 256), p256 = mt2 * up(N, 256);
    const bool pair128 = pairs > 0 && nkb >= 16 && mt2 * up(N, 128) <= pairs && mt * up(N, 64) > sms;
    if (t128 < sms) return pair128 ? TC_PAIR128 : TC_NARROW;
    const long w128 = up(t128, sms), ww = up(wide, sms), w256 = pairs > 0 ? up(p256, pairs) : 0;
    if (N >= 256 && f32) {
        if (w256 > 0 && w256 < w128) return TC_PAIR256;
        if (!pair128 && w128 == 2 && ww == 1) return TC_WIDE;
    } else if (N >= 256) {
        // [argmax][two chunks of K][pair256, wide, 128 x 128] {t, a, b, c}
        static constexpr double fit[2][2][3][4] = {
            {{{4.69, 0.162, 3.69, 0.116}, {3.09, 0.153, 4.24, 0.125}, {3.24, 0.137, 2.41, 0.142}},
             {{6.78, -0.026, 5.19, 0.206}, {3.99, -0.073, 11.89, 0.053}, {4.53, 0.015, 4.32, 0.149}}},
            {{{4.24, 0.138, 3.21, 0.139}, {2.89, 0.215, 4.82, 0.064}, {3.11, 0.150, 2.55, 0.133}},
             {{6.88, -0.034, 4.62, 0.214}, {4.09, -0.058, 12.17, 0.041}, {5.90, -0.030, 3.03, 0.193}}}};
        const auto time = [&](int v, long w) {
            const double *c = fit[argmax][nkb > 16][v];
            return c[0] + c[1] * nkb + (double)w * (c[2] + c[3] * nkb);
        };
        const double tp = time(0, w256), tw = time(1, ww), t1 = time(2, w128);
        if (w256 > 0 && (!rows16 || (tp < 0.97 * t1 && tp < (nkb > 8 ? 1.0 : 1.03) * tw))) return TC_PAIR256;
        if (!pair128 && tw < 0.97 * t1) return TC_WIDE;
    }
    return pair128 ? TC_PAIR128 : TC_128;
}

// LayerNorm of M rows of d: a warp per row (whole float4s, up to 1024 elements) or
// a block per row?  A warp per row from two rows per SM on, from three where the
// block kernel divides d among its threads without remainder (us, block / warp:
// 301 x 384 3.8 / 3.1, 301 x 512 2.75 / 3.2, 400 x 512 3.1 / 3.1, 512 x 512 3.6 / 3.2, 301 x 1024,
// codes only 3.6 / 4.4, 512 x 1024 4.9 / 4.5, 16384 x 512 38.1 / 20.6).
inline bool route_layernorm_warp(int M, int d) {
    return d % 4 == 0 && d <= 1024 && M > (d == 512 || d == 1024 ? 448 : 300);
}

// Fake quantisation of n elements: groups of 4 (forward) or 8 (backward) per
// thread and step, or single elements, and the blocks of 256 threads for it.
//   Single elements where an array is not 16-byte aligned, and where groups would
//   leave too few threads: a step's chain is then longer than its loads are worth
//   (us, single / groups: forward 10007 1.56 / 1.70, 65536 1.66 / 1.60; backward 100
//   7.1 / 8.2, 65536 8.9 / 8.7; min-max form 65536 8.7 / 10.3, 300000 11.6 / 11.0).
struct FqLaunch {
    bool groups;
    int blocks;
};
inline FqLaunch route_fake_quant(size_t n, bool aligned, bool backward, bool minmax, int sms) {
    FqLaunch l;
    l.groups = aligned && n >= (size_t)(!backward ? 32768 : minmax ? 262144 : 4096);
    const size_t per = l.groups ? (backward ? 8 : 4) : 1, b = (n / per + 255) / 256, cap = (size_t)8 * sms;
    l.blocks = (int)(b < 1 ? 1 : b > cap ? cap : b);
    return l;
}

// May the batched decode step run on `clusters` clusters of 8 nb rows with hpc
// heads per CTA, of which `fit` are resident at once?  (Tried with 1, 2 and 4
// times 8 rows of one head per CTA, then 16 rows of two; else a kernel per
// operation.)  A second wave of clusters doubles the step; 32 rows, or two heads,
// to a warp's chain are worth it only where beams share their keys.  Steps of
// 24, us, batched / kernel per operation:
//   one wave of 8 or 16 rows: d 128, 480 rows 66 / 95; d 256, 576 rows 110 / 128; d 512,
//     6 layers, 240 rows 205 / 251
//   32 rows: d 512, 400 rows, beam 1 267 / 229, beam 4 279 / 278; d 256, beam 4,
//     640 rows 203 / 197, 1152 rows 251 / 253; d 384, beam 4, 640 rows 154 / 163
//   16 rows of two heads: d 512, 576 rows, beam 1 281 / 267, beam 2 306 / 311, beam 4
//     293 / 314; steps of 128, beam 2, 444 rows 342 / 309, beam 4, 576 rows 318 / 353
//   32 rows of two heads: d 512, beam 4, 640 rows 404 / 324, beam 1 427 / 274
//   two waves: d 512, beam 1, 1200 rows 805 / 348
inline bool route_rows_variant(int nb, int hpc, int beam, int clusters, int fit) {
    return clusters <= fit && ((nb <= 2 && hpc == 1) || beam >= 4);
}

}  // namespace mnmt
