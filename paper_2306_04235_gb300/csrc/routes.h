// routes.h -- which kernel a call of several takes, by its sizes: plain host
// functions, so that the rules can be compared with measured times anywhere.
#pragma once

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
