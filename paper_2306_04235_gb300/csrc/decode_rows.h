// decode_rows.h -- the batched decode step's parameter block and launchers
// (decode_rows.cu).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace mnmt {

// ---- decode step of larger batches: clusters of H / hpc CTAs (hpc heads each), 8 nb rows each ----
constexpr int DR_LMAX = 16;  // decoder layers
constexpr int DR_FORMS[4][2] = {{1, 1}, {2, 1}, {4, 1}, {2, 2}};  // nb, hpc in the order of preference
struct DrLin {
    const float *s, *b, *inv;  // inv: requantisation constants (or null)
    float sx, gam;             // input scale; residual gain (W_o, W_2)
};
struct DrLayer {
    const float *ln1_g, *ln1_b, *ln2_g, *ln2_b, *ln3_g, *ln3_b;
    float inv_in1, inv_in2, inv_in3, sigma1, rho1, sigma2, rho2;
    DrLin lin[6];  // qkv, o, q2, o2, w1, w2
    int8_t *self_k, *self_v;          // [R][H][T][64]
    const int8_t *cross_k, *cross_v;  // [B][H][S][64]
};
struct alignas(16) DrParams {
    int R, d, H, F, E, V, T, S, n_dec, beam;
    const uint8_t *stream;  // packed weights [nc][stream_cta]
    size_t stream_cta;
    const int8_t *emb_q, *proj_w;  // proj_w: factorised E -> d (or null)
    const float *emb_s, *proj_s, *proj_b, *pe;
    float emb_scale, inv_dout;
    const float *fin_g, *fin_b;
    const int32_t *tok, *src_len, *anc;
    const int *t_ptr, *done;
    int8_t *act_out;
    __half *act16_out;  // or null
    float *resid_out;
    int *status;
    // shared-memory carve-up and constants filled by dr_layout
    int far_caches;  // the decoder's caches exceed L2
    int nc, param_bytes, cap, stride_a, stride_h, slots;
    int off_bar, off_a, off_h, off_y, off_r, off_q, off_red, off_stage, off_prow, off_meta, off_ln, off_ring;
    int ln_w, ln_epl, ln_kd, ln_dodd;  // log2 warps per row, elements per lane; d = ln_dodd 2^ln_kd
    unsigned long long ln_zm;
    DrLayer layer[DR_LMAX];
};
bool dr_shape_ok(int d, int H, int F, int E, int n_dec);
size_t dr_bytes(int d, int F, int n_dec);  // packed weights, all CTAs
struct DrPack {
    const int8_t *w[DR_LMAX][6];  // [N][K] codes of every decoder linear, in phase order
    int n_dec;
};
cudaError_t dr_pack(const DrPack &pk, int d, int H, int hpc, int F, uint8_t *out, cudaStream_t st);
size_t dr_layout(DrParams &P, int nb, int hpc, size_t max_smem);  // bytes of one CTA, or (size_t)-1
int dr_max_clusters(int nb, int hpc, int nc, size_t smem);        // clusters resident at once
cudaError_t decode_rows_init();
cudaError_t launch_decode_rows(const DrParams *dP, int nb, int hpc, int nc, int clusters, size_t smem, cudaStream_t st);

}  // namespace mnmt
