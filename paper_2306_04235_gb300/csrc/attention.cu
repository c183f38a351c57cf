// attention.cu -- scaled dot-product attention of the INT8 encoder-decoder
// (App. A, Eq. 1/2) per head, with the quantisation points of Fig. 5b: int8 Q,
// K, V and context; the softmax in full precision.
//
// Per head and query row: scores acc_j = q . k_j (exact int32, dp4a),
// s_j = fl(acc_j * sigma), m = max_j s_j, weights E_j = rne(exp(fl(s_j - m)) 2^24)
// (an integer in [0, 2^24]), context N_e = sum_j E_j v_j[e] and Z = sum_j E_j as
// exact integer sums (so any summation order gives the same bits), then
// ctx_e = q8(nearest fp32 to N_e / Z, rho).
//
// Kernels:
//   attn_decode  one warp per (row, head): the incremental step of the decoder
//                over the self-attention cache (keys 0..t, through the beam
//                ancestry table when hypotheses were reordered) or over the
//                cross-attention keys of the row's sentence.  Bound by the
//                cache bytes it streams.
//   attn_encoder one block per (sentence, head, chunk of 4..32 queries): K and V of
//                the head staged in shared memory, keys masked past the
//                source length (small grids, and d_h = 128).
//   attn_encoder_tc  the same for d_h = 32 and 64 on the tensor cores (mma.sync
//                on fp16 integers, exact): one block per (sentence, head,
//                16..64 queries).
#include <type_traits>

#include "attn_core.cuh"
#include "common.cuh"
#include "internal.h"

namespace mnmt {

constexpr int DEC_MAX_KEYS = 1024;

struct DecRows {
    const int8_t *kc, *vc;  // layer cache
    const int *prow;        // [n] physical row of every position (null: all `row`)
    int row, H, h, T, dh;
    MNMT_DEV size_t at(int j) const { return (((size_t)(prow ? prow[j] : row) * H + h) * T + j) * dh; }
    MNMT_DEV const int8_t *k(int j) const { return kc + at(j); }
    MNMT_DEV const int8_t *v(int j) const { return vc + at(j); }
};

// XS = false: a warp per (row, head).  XS = true (cross attention with beams):
// a warp per head and four of a sentence's beams, which read the same keys and
// values once.  LONGK: more than 512 keys may be attended (self attention only).
// Warps are independent, in blocks of four, MB of them to an SM: what bounds it
// is the loads in flight, and whether the grid fits at once.
// 512 rows x 8 heads of 64, 160 keys (84 MB): 28.0 us with whole rows per block,
// 26.2 in two waves of 24 warps per SM (6 blocks of 80 registers), 21.3 in one of
// 28 (7 of 72); 8 of 64 spill, 22.0.  80 keys: 17.8, 17.3, 13.8.  Grids that 24
// warps per SM hold prefer the registers (256 x 8, 500 of 512 keys: 56.4, 38.2,
// 39.1).  A key read by DH / 16 lanes instead of one: 512 x 4 heads of 128, 120
// keys 21.2 -> 17.4; of 64, 1 to 6 %.
constexpr int DEC_WARPS = 4;

template <int DH, bool XS, bool LONGK, int MB>
__global__ void __launch_bounds__(32 * DEC_WARPS, MB) attn_decode(AttnDecArgs a) {
    pdl_grid_wait();
    if (a.skip && *a.skip) return;
    constexpr int NB = XS ? 4 : 1;
    extern __shared__ __align__(16) int dsm[];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int item = blockIdx.x * DEC_WARPS + w, h = item % a.H;
    const int groups = XS ? (a.beam + NB - 1) / NB : 1;
    const int set = item / a.H;                          // row, or (sentence, four of its beams)
    const int b0 = XS ? set % groups * NB : 0;
    const int r = XS ? set / groups * a.beam + b0 : set;
    if (r >= a.R) return;
    const int nb = XS ? min(NB, a.beam - b0) : 1;
    int n, t = 0;
    if (a.cross) {
        n = a.src_len[r / a.beam];
        n = n < 1 ? 1 : (n > a.T ? a.T : n);  // lengths are validated on the host path; clamp on the device path
    } else if (a.n_keys) {
        n = a.n_keys[r];
        t = n - 1;
    } else {
        t = *a.t_ptr;
        n = t + 1;
    }
    const int cap = (a.T + 15) & ~15;  // key capacity: cache length / padded source length
    const bool gather = !XS && !a.cross && a.anc;  // positions live in other rows' caches
    int *sc = dsm + w * (NB + (gather ? 1 : 0)) * cap;  // this warp's [NB][cap] scores, then weights
    int *prow = sc + NB * cap;                          // [cap] physical row of every key position
    if (gather) {
        for (int j = lane; j < n; j += 32) prow[j] = j < t ? a.anc[(size_t)r * a.T + j] : r;
        __syncwarp();
    }
    const DecRows rows{a.kc, a.vc, gather ? prow : nullptr, a.cross ? r / a.beam : r, a.H, h, a.T, DH};
    const int d = a.H * DH;
    attn_rows<DH, NB, LONGK>(
        a.q + (size_t)r * d + h * DH, d, nb, n, a.sigma, a.rho, sc, cap, rows, [&](int b, int e, const uint32_t (&words)[DH / 32]) {
            const size_t o = (size_t)(r + b) * d + h * DH + e;
            const bool al = (reinterpret_cast<uintptr_t>(a.ctx) & 3) == 0;
#pragma unroll
            for (int i = 0; i < DH / 32; i++) {
                if (al) {
                    reinterpret_cast<uint32_t *>(a.ctx + o)[i] = words[i];
                } else {
#pragma unroll
                    for (int k = 0; k < 4; k++) a.ctx[o + 4 * i + k] = (int8_t)(words[i] >> (8 * k));
                }
                if (a.ctx16) {
                    uint32_t lo, hi;
                    codes_to_half2((int)words[i], lo, hi);
                    reinterpret_cast<uint32_t *>(a.ctx16 + o)[2 * i] = lo;
                    reinterpret_cast<uint32_t *>(a.ctx16 + o)[2 * i + 1] = hi;
                }
            }
        });
}

cudaError_t launch_attention_decode(const AttnDecArgs &a, cudaStream_t st) {
    if (a.H > 16 || a.T < 1 || a.T > DEC_MAX_KEYS) return cudaErrorInvalidValue;
    // cross attention with beams: a sentence's beams share a warp when there are
    // sentences enough for half of the SMs (with fewer, a warp per beam keeps
    // more SMs busy)
    const bool xs = a.cross && a.T <= ATT_CORE_MAX_KEYS && a.beam > 1 && a.R % a.beam == 0 &&
                    2 * (a.R / a.beam) >= device_sm_count();
    const long items = (long)a.H * (xs ? (a.R / a.beam) * ((a.beam + 3) / 4) : a.R);
    const size_t smem = (size_t)DEC_WARPS * (xs ? 4 : !a.cross && a.anc ? 2 : 1) * ((a.T + 15) & ~15) * sizeof(int);
    const dim3 block(32 * DEC_WARPS);
    const int grid = (int)((items + DEC_WARPS - 1) / DEC_WARPS);
    auto go = [&](auto dh) {
        constexpr int DH = decltype(dh)::value;
        constexpr int MB = DH == 128 ? 4 : 6, MANY = DH == 128 ? 4 : 7;
        if (xs) launch_pdl(attn_decode<DH, true, false, 4>, grid, block, smem, st, a);
        else if (a.T > ATT_CORE_MAX_KEYS) launch_pdl(attn_decode<DH, false, true, 4>, grid, block, smem, st, a);
        else if (grid > MB * device_sm_count()) launch_pdl(attn_decode<DH, false, false, MANY>, grid, block, smem, st, a);
        else launch_pdl(attn_decode<DH, false, false, MB>, grid, block, smem, st, a);
        return cudaGetLastError();
    };
    switch (a.dh) {
        case 32: return go(std::integral_constant<int, 32>{});
        case 64: return go(std::integral_constant<int, 64>{});
        case 128: return go(std::integral_constant<int, 128>{});
        default: return cudaErrorInvalidValue;
    }
}

// ---------------------------------------------------------------------------
// encoder self-attention
// ---------------------------------------------------------------------------
constexpr int ENC_WARPS = 4;
constexpr int ENC_MAX_KEYS = 512;
constexpr int ENC_QCHUNK = 32;

template <int DH>
__global__ void __launch_bounds__(32 * ENC_WARPS) attn_encoder(AttnEncArgs a, int qchunk) {
    pdl_grid_wait();
    extern __shared__ __align__(16) uint8_t esm[];
    constexpr int KS = DH + 16;  // padded key row: conflict-free 16-byte lane reads
    const int bh = blockIdx.x;
    const int b = bh / a.H, h = bh - b * a.H;
    const int S = a.S;
    int len = a.len[b];
    len = len < 1 ? 1 : (len > S ? S : len);  // validated on the host path; clamp on the device path
    uint8_t *Ks = esm;                         // [S][KS]
    int8_t *Vs = reinterpret_cast<int8_t *>(esm + (size_t)S * KS);  // [S][DH]
    int *wsm = reinterpret_cast<int *>(esm + (size_t)S * KS + (size_t)S * DH);  // [warps][S]
    const int ld = 3 * a.d;
    const int8_t *base = a.qkv + (size_t)b * S * ld;
    // stage K and V of this head (valid keys only)
    constexpr int CH = DH / 16;
    for (int i = threadIdx.x; i < len * CH; i += blockDim.x) {
        int j = i / CH, c = i - j * CH;
        const int4 *src = reinterpret_cast<const int4 *>(base + (size_t)j * ld + a.d + h * DH);
        reinterpret_cast<int4 *>(Ks + (size_t)j * KS)[c] = src[c];
        const int4 *vsrc = reinterpret_cast<const int4 *>(base + (size_t)j * ld + 2 * a.d + h * DH);
        reinterpret_cast<int4 *>(Vs + (size_t)j * DH)[c] = vsrc[c];
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int *sc = wsm + warp * S;
    const int q0 = blockIdx.y * qchunk;
    const int q1 = min(q0 + qchunk, S);
    constexpr int EPL = DH / 32;
    for (int qi = q0 + warp; qi < q1; qi += ENC_WARPS) {
        int4 qv[CH];
        const int4 *qp = reinterpret_cast<const int4 *>(base + (size_t)qi * ld + h * DH);
#pragma unroll
        for (int c = 0; c < CH; c++) qv[c] = qp[c];
        float mx = -INFINITY;
        for (int j = lane; j < len; j += 32) {
            const int4 *kr = reinterpret_cast<const int4 *>(Ks + (size_t)j * KS);
            int acc = 0;
#pragma unroll
            for (int c = 0; c < CH; c++) acc = dot16(qv[c], kr[c], acc);
            float s = __fmul_rn(__int2float_rn(acc), a.sigma);
            sc[j] = __float_as_int(s);
            mx = fmaxf(mx, s);
        }
        mx = warp_max_f(mx);
        long long Z = 0;
        for (int j = lane; j < len; j += 32) {
            int E = softmax_weight(__fadd_rn(__int_as_float(sc[j]), -mx));
            sc[j] = E;
            Z += E;
        }
        Z = warp_sum_ll(Z);
        __syncwarp();
        int hi[EPL], lo[EPL];
#pragma unroll
        for (int u = 0; u < EPL; u++) hi[u] = lo[u] = 0;
        for (int j = 0; j < len; j++) {
            int E = sc[j];
            int Eh = E >> 12, El = E & 4095;
            const int8_t *vr = Vs + (size_t)j * DH + lane * EPL;
#pragma unroll
            for (int u = 0; u < EPL; u++) {
                int v = vr[u];
                hi[u] += Eh * v;
                lo[u] += El * v;
            }
        }
        const size_t o = ((size_t)b * S + qi) * a.d + h * DH + lane * EPL;
        const float iz = softmax_inv(ll2float(Z));
#pragma unroll
        for (int u = 0; u < EPL; u++) {
            const int8_t v = q8_context_hl(hi[u], lo[u], iz, a.rho, [&]() {
                return att_ctx_exact((long long)hi[u] * 4096 + lo[u], Z, a.rho);
            });
            a.ctx[o + u] = v;
            if (a.ctx16) a.ctx16[o + u] = __short2half_rn(v);
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// encoder self-attention on the tensor cores (mma.sync m16n8k16, fp16 operands,
// fp32 accumulation), d_h = 32 or 64.  Same integers as attn_encoder: codes and
// weight pieces are fp16 integers, and every sum stays within 2^24, so fp32
// holds it exactly in any order.
//   scores   q . k_j: 64 products of at most 2^14.
//   context  E_j in [0, 2^24] is split into bytes, E_j = e0 + 2^8 e1 + 2^16 e2
//            with e2 <= 256; each sum_j e_kj v_j[e] is at most
//            512 * 256 * 128 = 2^24.
// The fp16 form is used because the int8 one is slow on this part: mma.sync s8
// measures 542 operations per clock and SM, f16 2048.
//
// One block of four warps per (sentence, head, 16 NW queries): all stage, NW
// compute, 16 queries each.  K and V are staged once per block as fp16 rows of 2 DH bytes, 16-byte chunks
// XOR-swizzled by row (ldmatrix without bank conflicts; .trans for V).  The
// scores are computed twice, for the row maximum and for the weights, which
// keeps them out of registers; the weights' accumulator fragments are the
// A fragments of the context products, so they never leave the registers.
// Bound by issue slots (exp and the byte split), then the tensor pipe.
// 64 x 100 tokens, 8 heads of 64: 101 us as four int8 products with the weight
// bytes in shared memory, 31 us so (ncu, cold).
// ---------------------------------------------------------------------------
MNMT_DEV uint32_t att_smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
MNMT_DEV void att_ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
MNMT_DEV void att_ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
// byte offset of (row, 16-byte chunk) in rows of 2 DH bytes
template <int DH>
MNMT_DEV int att_sw(int row, int chunk) {
    return DH == 64 ? row * 128 + ((chunk ^ (row & 7)) << 4) : row * 64 + ((chunk ^ ((row >> 1) & 3)) << 4);
}

constexpr int ENC_TC_THREADS = 128;
constexpr long ENC_TC_MIN_TILES = 192;

template <int DH, int NW>
__global__ void __launch_bounds__(ENC_TC_THREADS) attn_encoder_tc(AttnEncArgs a, int Sp) {
    pdl_grid_wait();
    extern __shared__ __align__(128) uint8_t emm[];
    constexpr int CH = DH / 16;        // 16-code chunks of an int8 row
    constexpr int KS = DH / 16;        // k-steps of the score product
    constexpr int NT = DH / 8;         // 8-column tiles of the context
    constexpr int RB = 2 * DH;         // bytes of an fp16 row
    const int bh = blockIdx.x;
    const int b = bh / a.H, h = bh - b * a.H;
    const int S = a.S;
    int len = a.len[b];
    len = len < 1 ? 1 : (len > S ? S : len);  // validated on the host path; clamp on the device path
    const int lp = (len + 15) & ~15;          // keys the products run over
    const int q0 = blockIdx.y * (16 * NW);
    uint8_t *Qs = emm;                         // [16 NW][DH] fp16, then the output rows
    uint8_t *Ks = Qs + 16 * NW * RB;           // [Sp][DH] fp16
    uint8_t *Vs = Ks + (size_t)Sp * RB;        // [Sp][DH] fp16
    const int ld = 3 * a.d;
    const int8_t *base = a.qkv + (size_t)b * S * ld + h * DH;
    auto put16 = [&](uint8_t *rows, int r, int c, const int4 v) {
        uint32_t o[8];
        codes_to_half2(v.x, o[0], o[1]);
        codes_to_half2(v.y, o[2], o[3]);
        codes_to_half2(v.z, o[4], o[5]);
        codes_to_half2(v.w, o[6], o[7]);
        *reinterpret_cast<uint4 *>(rows + att_sw<DH>(r, 2 * c)) = make_uint4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<uint4 *>(rows + att_sw<DH>(r, 2 * c + 1)) = make_uint4(o[4], o[5], o[6], o[7]);
    };
    const int4 zero = make_int4(0, 0, 0, 0);
    for (int i = threadIdx.x; i < 16 * NW * CH; i += ENC_TC_THREADS) {
        const int r = i / CH, c = i % CH, q = q0 + r;
        put16(Qs, r, c, q < S ? reinterpret_cast<const int4 *>(base + (size_t)q * ld)[c] : zero);
    }
#pragma unroll 2
    for (int i = threadIdx.x; i < lp * CH; i += ENC_TC_THREADS) {
        const int j = i / CH, c = i % CH;
        int4 kv = zero, vv = zero;
        if (j < len) {
            kv = reinterpret_cast<const int4 *>(base + (size_t)j * ld + a.d)[c];
            vv = reinterpret_cast<const int4 *>(base + (size_t)j * ld + 2 * a.d)[c];
        }
        put16(Ks, j, c, kv);
        put16(Vs, j, c, vv);
    }
    __syncthreads();

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp >= NW || q0 + warp * 16 >= S) return;
    const int jq = lane >> 3, i8 = lane & 7, g = lane >> 2, tq = lane & 3;
    uint32_t af[KS][4];
#pragma unroll
    for (int kk = 0; kk < KS; kk++)
        att_ldmatrix_x4(af[kk], att_smem_u32(Qs + att_sw<DH>(warp * 16 + (jq & 1) * 8 + i8, kk * 2 + (jq >> 1))));
    // scores of 16 keys: exact integers, then fl(acc sigma), -inf past the source length
    auto scores16 = [&](int k0, float (&sv)[2][4]) {
        float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
        for (int kk = 0; kk < KS; kk++) {
            uint32_t r[4];
            att_ldmatrix_x4(r, att_smem_u32(Ks + att_sw<DH>(k0 + (jq >> 1) * 8 + i8, kk * 2 + (jq & 1))));
            mma_f16_16816(acc[0], af[kk], r[0], r[1]);
            mma_f16_16816(acc[1], af[kk], r[2], r[3]);
        }
#pragma unroll
        for (int t = 0; t < 2; t++)
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int key = k0 + t * 8 + tq * 2 + (q & 1);
                sv[t][q] = key < len ? __fmul_rn(acc[t][q], a.sigma) : -INFINITY;
            }
    };
    float mx0 = -INFINITY, mx1 = -INFINITY;  // rows g and g + 8
    for (int k0 = 0; k0 < lp; k0 += 16) {
        float sv[2][4];
        scores16(k0, sv);
#pragma unroll
        for (int t = 0; t < 2; t++) {
            mx0 = fmaxf(mx0, fmaxf(sv[t][0], sv[t][1]));
            mx1 = fmaxf(mx1, fmaxf(sv[t][2], sv[t][3]));
        }
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        mx0 = fmaxf(mx0, __shfl_xor_sync(0xFFFFFFFFu, mx0, o));
        mx1 = fmaxf(mx1, __shfl_xor_sync(0xFFFFFFFFu, mx1, o));
    }
    // weights (the scores again), their bytes as fp16 A fragments, the context products
    uint32_t z0 = 0, z1 = 0;  // at most 128 weights of 2^24 per lane
    float acc[3][NT][4];
#pragma unroll
    for (int L = 0; L < 3; L++)
#pragma unroll
        for (int nt = 0; nt < NT; nt++)
#pragma unroll
            for (int q = 0; q < 4; q++) acc[L][nt][q] = 0.0f;
#pragma unroll 1
    for (int k0 = 0; k0 < lp; k0 += 16) {
        float sv[2][4];
        scores16(k0, sv);
        uint32_t E[2][4];
#pragma unroll
        for (int t = 0; t < 2; t++) {
#pragma unroll
            for (int q = 0; q < 4; q++)
                E[t][q] = (uint32_t)softmax_weight(__fsub_rn(sv[t][q], q < 2 ? mx0 : mx1));
            z0 += E[t][0] + E[t][1];
            z1 += E[t][2] + E[t][3];
        }
        uint32_t vb[NT / 2][4];
#pragma unroll
        for (int nj = 0; nj < NT / 2; nj++)
            att_ldmatrix_x4_trans(vb[nj],
                                  att_smem_u32(Vs + att_sw<DH>(k0 + (jq & 1) * 8 + i8, 2 * nj + (jq >> 1))));
#pragma unroll
        for (int L = 0; L < 3; L++) {
            // byte L (byte pair of e2, up to 256) of two weights as fp16: 0x6400 | n is 1024 + n
            uint32_t ea[4];
#pragma unroll
            for (int f = 0; f < 4; f++) {
                const uint32_t lo = E[f >> 1][2 * (f & 1)], hi = E[f >> 1][2 * (f & 1) + 1];
                const uint32_t w = L == 2 ? __byte_perm(lo, hi, 0x7632) : __byte_perm(lo, hi, L ? 0x6521 : 0x5410);
                ea[f] = half2_sub_1024((w & (L == 2 ? 0x01FF01FFu : 0x00FF00FFu)) | 0x64006400u);
            }
#pragma unroll
            for (int nj = 0; nj < NT / 2; nj++) {
                mma_f16_16816(acc[L][2 * nj], ea, vb[nj][0], vb[nj][1]);
                mma_f16_16816(acc[L][2 * nj + 1], ea, vb[nj][2], vb[nj][3]);
            }
        }
    }
    long long Z0 = z0, Z1 = z1;
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        Z0 += __shfl_xor_sync(0xFFFFFFFFu, Z0, o);
        Z1 += __shfl_xor_sync(0xFFFFFFFFu, Z1, o);
    }
    // N = a0 + 2^8 a1 + 2^16 a2: fl(2^8 a1 + a0) is off by at most 2^8 + 1, which
    // makes at most rho 2^-15 of t (Z >= 2^24)
    const float iz0 = softmax_inv(ll2float(Z0)), iz1 = softmax_inv(ll2float(Z1));
    const float slack = __fmul_rn(fabsf(a.rho), 0x1p-15f);
    uint8_t *Os = Qs + warp * 16 * RB;  // this warp's own query rows: the output as fp16
    __syncwarp();
#pragma unroll
    for (int nt = 0; nt < NT; nt++)
#pragma unroll
        for (int hr = 0; hr < 2; hr++) {
            float c[2];
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const float a0 = acc[0][nt][2 * hr + q], a1 = acc[1][nt][2 * hr + q], a2 = acc[2][nt][2 * hr + q];
                const float fn = __fmaf_rn(a2, 65536.0f, __fmaf_rn(a1, 256.0f, a0));
                c[q] = q8_context(fn, hr ? iz1 : iz0, a.rho, slack, [&]() {
                    return att_ctx_exact((long long)__float2int_rn(a0) + (long long)__float2int_rn(a1) * 256 +
                                             (long long)__float2int_rn(a2) * 65536,
                                         hr ? Z1 : Z0, a.rho);
                });
            }
            const __half2 hv = __floats2half2_rn(c[0], c[1]);
            *reinterpret_cast<__half2 *>(Os + att_sw<DH>(g + 8 * hr, nt) + tq * 4) = hv;
        }
    __syncwarp();
    // rows of 16 codes per lane: fp16 as they are, int8 from the low byte of 1536 + v
    for (int i = lane; i < 16 * CH; i += 32) {
        const int r = i / CH, c = i % CH, qrow = q0 + warp * 16 + r;
        if (qrow >= S) continue;
        const uint4 lo = *reinterpret_cast<const uint4 *>(Os + att_sw<DH>(r, 2 * c));
        const uint4 hi = *reinterpret_cast<const uint4 *>(Os + att_sw<DH>(r, 2 * c + 1));
        const size_t o = ((size_t)b * S + qrow) * a.d + h * DH + 16 * c;
        *reinterpret_cast<uint4 *>(a.ctx + o) = make_uint4(half2_to_codes(lo.x, lo.y), half2_to_codes(lo.z, lo.w),
                                                           half2_to_codes(hi.x, hi.y), half2_to_codes(hi.z, hi.w));
        if (a.ctx16) {
            reinterpret_cast<uint4 *>(a.ctx16 + o)[0] = lo;
            reinterpret_cast<uint4 *>(a.ctx16 + o)[1] = hi;
        }
    }
}

template <int DH>
static size_t enc_tc_smem(int S, int nw) { return (size_t)(16 * nw + 2 * ((S + 15) & ~15)) * 2 * DH; }

template <int DH>
static cudaError_t launch_enc(const AttnEncArgs &a, cudaStream_t st) {
    size_t smem = (size_t)a.S * (DH + 16) + (size_t)a.S * DH + (size_t)ENC_WARPS * a.S * sizeof(int);
    auto k = attn_encoder<DH>;
    // queries per block: the most (up to 32) that still gives every SM two
    // blocks; small batches get one query per warp so the GPU fills up
    int qc = ENC_QCHUNK;
    while (qc > ENC_WARPS && (long)a.B * a.H * ((a.S + qc - 1) / qc) < 2 * 152) qc >>= 1;
    dim3 grid(a.B * a.H, (a.S + qc - 1) / qc);
    launch_pdl(k, grid, 32 * ENC_WARPS, smem, st, a, qc);
    return cudaGetLastError();
}

template <int DH, int NW>
static cudaError_t launch_enc_tc_nw(const AttnEncArgs &a, cudaStream_t st) {
    const dim3 grid(a.B * a.H, (a.S + 16 * NW - 1) / (16 * NW));
    launch_pdl(attn_encoder_tc<DH, NW>, grid, ENC_TC_THREADS, enc_tc_smem<DH>(a.S, NW), st, a, (a.S + 15) & ~15);
    return cudaGetLastError();
}

// warps (16 queries each) per block: four share a staging of K and V; fewer
// when that would leave SMs without a block or hold warps without queries
template <int DH>
static cudaError_t launch_enc_tc(const AttnEncArgs &a, cudaStream_t st) {
    const int tiles = (a.S + 15) / 16;
    int nw = tiles >= 3 ? 4 : tiles;
    while (nw > 1 && (long)a.B * a.H * ((tiles + nw - 1) / nw) < device_sm_count()) nw >>= 1;
    if (nw == 4) return launch_enc_tc_nw<DH, 4>(a, st);
    if (nw == 2) return launch_enc_tc_nw<DH, 2>(a, st);
    return launch_enc_tc_nw<DH, 1>(a, st);
}

cudaError_t launch_attention_encoder(const AttnEncArgs &a, cudaStream_t st) {
    if (a.S < 1 || a.S > ENC_MAX_KEYS) return cudaErrorInvalidValue;
    // few 16-query tiles: the dp4a kernel, one query per warp, has the shorter
    // chain (encode of one 46-token sentence, 12 layers: 402 against 440 us;
    // equal at 192 tiles; 8 x 100 tokens, 224 tiles: 634 against 561 us)
    const bool tc = (long)a.B * a.H * ((a.S + 15) / 16) > ENC_TC_MIN_TILES;
    switch (a.dh) {
        case 32:
            return tc ? launch_enc_tc<32>(a, st) : launch_enc<32>(a, st);
        case 64:
            return tc ? launch_enc_tc<64>(a, st) : launch_enc<64>(a, st);
        case 128:
            return launch_enc<128>(a, st);
        default:
            return cudaErrorInvalidValue;
    }
}

}  // namespace mnmt

namespace mnmt {
// Opt the attention kernels into the shared memory their largest shapes use
// (called once per process before any launch or stream capture).
cudaError_t attention_init() {
    cudaError_t err = cudaSuccess;
    const int dec = DEC_WARPS * 2 * DEC_MAX_KEYS * (int)sizeof(int);
    const int xs = DEC_WARPS * 4 * ATT_CORE_MAX_KEYS * (int)sizeof(int);
    auto dec_attr = [&](auto k, int smem) {
        if (!err) err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    };
    dec_attr(attn_decode<32, false, false, 6>, dec);
    dec_attr(attn_decode<64, false, false, 6>, dec);
    dec_attr(attn_decode<32, false, false, 7>, dec);
    dec_attr(attn_decode<64, false, false, 7>, dec);
    dec_attr(attn_decode<128, false, false, 4>, dec);
    dec_attr(attn_decode<32, true, false, 4>, xs);
    dec_attr(attn_decode<64, true, false, 4>, xs);
    dec_attr(attn_decode<128, true, false, 4>, xs);
    dec_attr(attn_decode<32, false, true, 4>, dec);
    dec_attr(attn_decode<64, false, true, 4>, dec);
    dec_attr(attn_decode<128, false, true, 4>, dec);
    auto enc = [](int dh) { return ENC_MAX_KEYS * (dh + 16) + ENC_MAX_KEYS * dh + ENC_WARPS * ENC_MAX_KEYS * 4; };
    if (!err) err = cudaFuncSetAttribute(attn_encoder<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, enc(32));
    if (!err) err = cudaFuncSetAttribute(attn_encoder<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, enc(64));
    if (!err) err = cudaFuncSetAttribute(attn_encoder<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, enc(128));
    auto enc_tc = [&](auto k, size_t smem) {
        if (!err) err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    };
    enc_tc(attn_encoder_tc<32, 1>, enc_tc_smem<32>(ENC_MAX_KEYS, 1));
    enc_tc(attn_encoder_tc<32, 2>, enc_tc_smem<32>(ENC_MAX_KEYS, 2));
    enc_tc(attn_encoder_tc<32, 4>, enc_tc_smem<32>(ENC_MAX_KEYS, 4));
    enc_tc(attn_encoder_tc<64, 1>, enc_tc_smem<64>(ENC_MAX_KEYS, 1));
    enc_tc(attn_encoder_tc<64, 2>, enc_tc_smem<64>(ENC_MAX_KEYS, 2));
    enc_tc(attn_encoder_tc<64, 4>, enc_tc_smem<64>(ENC_MAX_KEYS, 4));
    return err;
}
}  // namespace mnmt
