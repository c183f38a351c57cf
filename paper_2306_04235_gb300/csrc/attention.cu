// attention.cu -- scaled dot-product attention of the INT8 encoder-decoder
// (App. A, Eq. 1/2) per head, with the quantisation points of Fig. 5b: int8 Q,
// K, V and context; the softmax in full precision.
//
// Per head and query row: scores acc_j = q . k_j (exact int32, dp4a),
// s_j = fl(acc_j * sigma), m = max_j s_j, weights E_j = rne(exp(fl(s_j - m)) 2^24)
// (an integer in [0, 2^24]), context N_e = sum_j E_j v_j[e] and Z = sum_j E_j as
// exact integer sums (so any summation order gives the same bits), then
// ctx_e = q8(nearest fp32 to N_e / Z, rho).  N_e is accumulated in two int32 halves,
// E_j = Eh 2^12 + El, which cannot overflow for up to 1024 keys.
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

#include "common.cuh"
#include "internal.h"

namespace mnmt {

constexpr int DEC_MAX_KEYS = 1024;

// 32-bit word k of a 4-, 8- or 16-byte vector held in registers
MNMT_DEV uint32_t vec_word(uint32_t v, int) { return v; }
MNMT_DEV uint32_t vec_word(const uint2 &v, int k) { return k ? v.y : v.x; }
MNMT_DEV uint32_t vec_word(const uint4 &v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }

// the exact form of a context code (q8_context's undecided values)
__device__ __noinline__ float att_ctx_exact(long long n, long long z, float rho) {
    return (float)q8(rn32_div(n, z), rho);
}

// XS = false: one block per row, one warp per head.  XS = true (cross
// attention with beams): one block per sentence, one warp per (beam, head) --
// the beams of a sentence read the same keys and values, which their block
// then fetches from L2 once and serves from L1.
template <int DH, bool XS>
__global__ void __launch_bounds__(XS ? 32 * 32 : 32 * 16) attn_decode(AttnDecArgs a) {
    pdl_grid_wait();
    if (a.skip && *a.skip) return;
    extern __shared__ int dsm[];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = XS ? blockIdx.x * a.beam + w / a.H : blockIdx.x;
    const int h = XS ? w % a.H : w;
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
    const int cap = a.T;  // key capacity: cache length / padded source length
    int *prow = dsm;      // [cap] physical row of every key position (shared by the heads of this row)
    int *sc = XS ? dsm + w * cap : dsm + cap + h * cap;  // per warp [cap]: scores, then weights
    if (!XS) {
        for (int j = threadIdx.x; j < n; j += blockDim.x) {
            int p;
            if (a.cross) p = r / a.beam;
            else p = (a.anc && j < t) ? a.anc[(size_t)r * a.T + j] : r;
            prow[j] = p;
        }
        __syncthreads();
        if (h >= a.H) return;
    }
    const int psent = r / a.beam;  // XS: the sentence of every key
    auto prow_of = [&](int j) { return XS ? psent : prow[j]; };

    constexpr int QC = DH / 16;
    int4 qv[QC];
    const int4 *qp = reinterpret_cast<const int4 *>(a.q + (size_t)r * a.H * DH + h * DH);
#pragma unroll
    for (int c = 0; c < QC; c++) qv[c] = qp[c];

    float mx = -INFINITY;
#pragma unroll 4
    for (int j = lane; j < n; j += 32) {
        const int4 *kr = reinterpret_cast<const int4 *>(a.kc + (((size_t)prow_of(j) * a.H + h) * a.T + j) * DH);
        int acc = 0;
#pragma unroll
        for (int c = 0; c < QC; c++) acc = dot16(qv[c], kr[c], acc);
        float s = __fmul_rn(__int2float_rn(acc), a.sigma);
        sc[j] = __float_as_int(s);
        mx = fmaxf(mx, s);
    }
    mx = warp_max_f(mx);
    long long Z = 0;
    for (int j = lane; j < n; j += 32) {
        int E = softmax_weight(__fadd_rn(__int_as_float(sc[j]), -mx));
        sc[j] = E;
        Z += E;
    }
    Z = warp_sum_ll(Z);
    __syncwarp();

    // context: the warp takes CG keys at a time, one per group of 8 lanes;
    // lane gl of a group holds EPG consecutive elements of the head, read as
    // one EPG-byte load per key.  N_e = sum_j E_j v_j[e] is split into 12-bit
    // halves of E_j so that every partial stays an exact int32.
    constexpr int CG = 4, LPG = 32 / CG, EPG = DH / LPG;
    using VecT = typename std::conditional<EPG == 4, uint32_t, typename std::conditional<EPG == 8, uint2, uint4>::type>::type;
    const int grp = lane / LPG, gl = lane % LPG;
    int hi[EPG], lo[EPG];
#pragma unroll
    for (int u = 0; u < EPG; u++) hi[u] = lo[u] = 0;
    auto vload = [&](int j) -> VecT {
        return *reinterpret_cast<const VecT *>(a.vc + (((size_t)prow_of(j) * a.H + h) * a.T + j) * DH + gl * EPG);
    };
    auto vacc = [&](int j, const VecT &raw) {
        const int E = sc[j];
        const int Eh = E >> 12, El = E & 4095;
#pragma unroll
        for (int u = 0; u < EPG; u++) {
            const int v = (int)(int8_t)(vec_word(raw, u >> 2) >> (8 * (u & 3)));
            hi[u] += Eh * v;
            lo[u] += El * v;
        }
    };
    // groups of UJ rounds: every value load of the batch is issued before any
    // is used, so their latencies overlap
    constexpr int UJ = DH == 128 ? 2 : 4;
    int j0 = 0;
    for (; j0 + CG * UJ <= n; j0 += CG * UJ) {
        VecT raw[UJ];
#pragma unroll
        for (int u = 0; u < UJ; u++) raw[u] = vload(j0 + u * CG + grp);
#pragma unroll
        for (int u = 0; u < UJ; u++) vacc(j0 + u * CG + grp, raw[u]);
    }
    for (int j = j0 + grp; j < n; j += CG) vacc(j, vload(j));
    // sum over the CG groups (lanes gl, gl+8, gl+16, gl+24): every lane gets the totals
#pragma unroll
    for (int u = 0; u < EPG; u++) {
#pragma unroll
        for (int o = LPG; o < 32; o <<= 1) {
            hi[u] += __shfl_xor_sync(0xFFFFFFFFu, hi[u], o);
            lo[u] += __shfl_xor_sync(0xFFFFFFFFu, lo[u], o);
        }
    }
    // lane (grp, gl) writes elements gl * EPG + grp * EPG / CG + [0, EPG / CG)
    constexpr int OPL = EPG / CG;
    const size_t o = (size_t)r * a.H * DH + h * DH + gl * EPG + grp * OPL;
#pragma unroll
    for (int u = 0; u < EPG; u++) {
        if (u / OPL == grp) {
            long long N = (long long)hi[u] * 4096 + lo[u];
            const int8_t v = q8_quotient(N, Z, a.rho, rn32_div);
            a.ctx[o + u - grp * OPL] = v;
            if (a.ctx16) a.ctx16[o + u - grp * OPL] = __short2half_rn(v);
        }
    }
}

cudaError_t launch_attention_decode(const AttnDecArgs &a, cudaStream_t st) {
    if (a.H > 16 || a.T < 1 || a.T > DEC_MAX_KEYS) return cudaErrorInvalidValue;
    // cross attention with beams: the beams of a sentence share a block, when
    // there are sentences enough for half of the SMs (measured on 152 SMs:
    // 3.8 us per step faster at 128 sentences, 1.7 us slower at 32)
    const bool xs = a.cross && a.beam > 1 && a.beam * a.H <= 32 && a.R % a.beam == 0 &&
                    2 * (a.R / a.beam) >= device_sm_count();
    const size_t smem = (size_t)(xs ? a.beam * a.H : 1 + a.H) * a.T * sizeof(int);
    const dim3 block(32 * a.H * (xs ? a.beam : 1));
    const int grid = xs ? a.R / a.beam : a.R;
    switch (a.dh) {
        case 32:
            if (xs) launch_pdl(attn_decode<32, true>, grid, block, smem, st, a);
            else launch_pdl(attn_decode<32, false>, grid, block, smem, st, a);
            break;
        case 64:
            if (xs) launch_pdl(attn_decode<64, true>, grid, block, smem, st, a);
            else launch_pdl(attn_decode<64, false>, grid, block, smem, st, a);
            break;
        case 128:
            if (xs) launch_pdl(attn_decode<128, true>, grid, block, smem, st, a);
            else launch_pdl(attn_decode<128, false>, grid, block, smem, st, a);
            break;
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
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
        const float iz = __frcp_rn(__ll2float_rn(Z));
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
    const float iz0 = __frcp_rn(__ll2float_rn(Z0)), iz1 = __frcp_rn(__ll2float_rn(Z1));
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
    int dec = (1 + 16) * DEC_MAX_KEYS * (int)sizeof(int);
    const int xs = 32 * DEC_MAX_KEYS * (int)sizeof(int);  // up to 32 (beam, head) warps
    if (!err) err = cudaFuncSetAttribute(attn_decode<32, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, dec);
    if (!err) err = cudaFuncSetAttribute(attn_decode<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, dec);
    if (!err) err = cudaFuncSetAttribute(attn_decode<128, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, dec);
    if (!err) err = cudaFuncSetAttribute(attn_decode<32, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, xs);
    if (!err) err = cudaFuncSetAttribute(attn_decode<64, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, xs);
    if (!err) err = cudaFuncSetAttribute(attn_decode<128, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, xs);
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
