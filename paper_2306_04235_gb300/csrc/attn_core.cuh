// attn_core.cuh -- incremental attention (Eq. 1/2, Fig. 5b) of up to four query
// rows of one head by one warp, keys and values read from int8 caches.
//
//   scores   acc = q . k by dp4a (exact int32), s = fl(acc sigma); a key is read
//            by DH / 16 lanes, 16 bytes each (a lane per key touched a line for
//            every 16 bytes), whose sums are scattered over them.
//   weights  E = rne(exp(s - max) 2^24) in [0, 2^24], kept in shared memory.
//   context  sum_j E_j v_j on the fp16 tensor cores (mma.sync m16n8k16, 16 keys
//            per step): E = e0 + 2^8 e1 + 2^16 e2 (e2 <= 256), the operand rows
//            are (byte, query row) pairs -- rows 0..3 and 4..7 the bytes e0 and
//            e1 of the four queries, rows 8..11 their e2 -- and the columns
//            elements of v.  Codes and bytes are fp16 integers; a sum over at
//            most 512 keys is at most 512 * 256 * 128 = 2^24, so fp32 holds every
//            partial sum exactly.  A lane reads whole words of four keys of its
//            step and turns them into operand registers with byte permutes.
// The integer form of the context (two multiply-adds per key and element, after
// extracting the byte) costs ~4 instructions per value and query against ~1.5 per
// value here, and its loads wait on one another more often.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "epilogue.cuh"

namespace mnmt {

constexpr int ATT_CORE_MAX_KEYS = 512;

// the exact form of a context code (q8_context's undecided values)
static __device__ __noinline__ float att_ctx_exact(long long n, long long z, float rho) {
    return (float)q8(rn32_div(n, z), rho);
}

// EPG consecutive bytes of a value row
template <int EPG>
struct AttVec {
    using T = typename std::conditional<EPG == 4, uint32_t, typename std::conditional<EPG == 8, uint2, uint4>::type>::type;
};
MNMT_DEV uint32_t att_word(uint32_t v, int) { return v; }
MNMT_DEV uint32_t att_word(const uint2 &v, int k) { return k ? v.y : v.x; }
MNMT_DEV uint32_t att_word(const uint4 &v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }

// rows.k(j), rows.v(j): the key / value row of position j, for every query row.
// q: [NB][q_ld] codes of the head (16-byte aligned rows), sc: this warp's
// [NB][cap] weights, cap a multiple of 16, at least n; n <= ATT_CORE_MAX_KEYS
// unless LONGK.
// store(b, e, words): EPG codes from element e of row b.
template <int DH, int NB, bool LONGK, typename Rows, typename Store>
__device__ __forceinline__ void attn_rows(const int8_t *q, int q_ld, int nb, int n, float sigma, float rho, int *sc, int cap,
                        const Rows &rows, const Store &store) {
    constexpr int LPK = DH / 16, KPL = 32 / LPK, EPG = DH / 8, NT = DH / 8;  // lanes per key, keys per load
    using Vec = typename AttVec<EPG>::T;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int kc = lane % LPK, kg = lane / LPK;
    float mx[NB];
    int4 qr[NB];
#pragma unroll
    for (int b = 0; b < NB; b++) {
        mx[b] = -INFINITY;
        qr[b] = *reinterpret_cast<const int4 *>(q + (size_t)(b < nb ? b : 0) * q_ld + 16 * kc);
    }
#pragma unroll 2
    for (int j0 = 0; j0 < n; j0 += 32) {
        int4 kr[LPK];
#pragma unroll
        for (int i = 0; i < LPK; i++) kr[i] = *reinterpret_cast<const int4 *>(rows.k(min(j0 + KPL * i + kg, n - 1)) + 16 * kc);
        const int j = j0 + KPL * kc + kg;  // the key whose sum this lane ends with
#pragma unroll
        for (int b = 0; b < NB; b++) {
            int acc[LPK];
#pragma unroll
            for (int i = 0; i < LPK; i++) acc[i] = dot16(qr[b], kr[i], 0);
            gemv_reduce<LPK, LPK>(acc, kc);
            if (j < n && b < nb) {
                const float s = __fmul_rn(__int2float_rn(acc[0]), sigma);
                sc[b * cap + j] = __float_as_int(s);
                mx[b] = fmaxf(mx[b], s);
            }
        }
    }
    __syncwarp();
    const int n16 = (n + 15) & ~15;
    long long Z[NB];
    float iz[NB];
#pragma unroll
    for (int b = 0; b < NB; b++) {
        Z[b] = 1;
        iz[b] = 0.0f;
        if (b > 0 && b >= nb) continue;
        const float m = warp_max_f(mx[b]);
        uint32_t z = 0;  // at most 32 weights of 2^24 per lane
        for (int j = lane; j < n16; j += 32) {
            const int E = j < n ? softmax_weight(__fsub_rn(__int_as_float(sc[b * cap + j]), m)) : 0;
            sc[b * cap + j] = E;
            z += (uint32_t)E;
        }
        Z[b] = warp_sum_exact((long long)z);
        iz[b] = softmax_inv(ll2float(Z[b]));
    }
    __syncwarp();

    float acc[NT][4];
#pragma unroll
    for (int j = 0; j < NT; j++)
#pragma unroll
        for (int i = 0; i < 4; i++) acc[j][i] = 0.0f;
    const int qb = g & 3;
    const int sh = g >= 4 ? 8 : 0;
    const uint32_t m01 = qb < nb ? 0x00FF00FFu : 0u, m2 = qb < nb && g < 4 ? 0x01FF01FFu : 0u;
    const int *er = sc + (qb < nb ? qb : 0) * cap + 4 * t;
    auto vload = [&](int kb, Vec (&raw)[4]) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int key = min(kb * 16 + 4 * t + i, n - 1);  // past the end: weight 0
            raw[i] = *reinterpret_cast<const Vec *>(rows.v(key) + EPG * g);
        }
    };
    auto step = [&](int kb, const Vec (&raw)[4]) {
        const int4 e = *reinterpret_cast<const int4 *>(er + kb * 16);
        uint32_t a[4];
        a[0] = half2_sub_1024((__byte_perm((uint32_t)e.x >> sh, (uint32_t)e.y >> sh, 0x5410) & m01) | 0x64006400u);
        a[2] = half2_sub_1024((__byte_perm((uint32_t)e.z >> sh, (uint32_t)e.w >> sh, 0x5410) & m01) | 0x64006400u);
        a[1] = half2_sub_1024((__byte_perm((uint32_t)e.x, (uint32_t)e.y, 0x7632) & m2) | 0x64006400u);
        a[3] = half2_sub_1024((__byte_perm((uint32_t)e.z, (uint32_t)e.w, 0x7632) & m2) | 0x64006400u);
#pragma unroll
        for (int w = 0; w < EPG / 4; w++) {
            uint32_t u[4], bq[4][2];
#pragma unroll
            for (int i = 0; i < 4; i++) u[i] = att_word(raw[i], w) ^ 0x80808080u;
#pragma unroll
            for (int p = 0; p < 2; p++) {  // keys (0, 1), then (2, 3) of this lane
                const uint32_t lo = __byte_perm(u[2 * p], u[2 * p + 1], 0x5140),
                               hi = __byte_perm(u[2 * p], u[2 * p + 1], 0x7362);
                bq[0][p] = h2_sub(__byte_perm(lo, 0x64646464u, 0x4140), 0x64806480u);
                bq[1][p] = h2_sub(__byte_perm(lo, 0x64646464u, 0x4342), 0x64806480u);
                bq[2][p] = h2_sub(__byte_perm(hi, 0x64646464u, 0x4140), 0x64806480u);
                bq[3][p] = h2_sub(__byte_perm(hi, 0x64646464u, 0x4342), 0x64806480u);
            }
#pragma unroll
            for (int x = 0; x < 4; x++) mma_f16_16816(acc[4 * w + x], a, bq[x][0], bq[x][1]);
        }
    };
    const int nkb = n16 >> 4;
    int tot[LONGK ? NT : 1][4];
    constexpr int UB = 2;  // steps whose loads are in flight together
    auto run = [&](int kb, int end) {
        for (; kb + UB <= end; kb += UB) {
            Vec raw[UB][4];
#pragma unroll
            for (int u = 0; u < UB; u++) vload(kb + u, raw[u]);
#pragma unroll
            for (int u = 0; u < UB; u++) step(kb + u, raw[u]);
        }
        for (; kb < end; kb++) {
            Vec raw[4];
            vload(kb, raw);
            step(kb, raw);
        }
    };
    if (!LONGK) {
        run(0, nkb);
    } else {
#pragma unroll
        for (int j = 0; j < NT; j++)
#pragma unroll
            for (int i = 0; i < 4; i++) tot[LONGK ? j : 0][i] = 0;
#pragma unroll 1
        for (int k0 = 0; k0 < nkb; k0 += ATT_CORE_MAX_KEYS / 16) {
            run(k0, min(nkb, k0 + ATT_CORE_MAX_KEYS / 16));
#pragma unroll
            for (int j = 0; j < NT; j++)
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    tot[LONGK ? j : 0][i] += __float2int_rn(acc[j][i]);
                    acc[j][i] = 0.0f;
                }
        }
#pragma unroll
        for (int j = 0; j < NT; j++)
#pragma unroll
            for (int i = 0; i < 4; i++) acc[j][i] = __int_as_float(tot[LONGK ? j : 0][i]);  // carried as bits
    }
    // lanes g < 4 finish the elements EPG 2 t + j of row g, lanes g >= 4 those
    // from EPG (2 t + 1) of row g - 4
    // (fl(2^8 a1 + a0) is off by at most 2^8 + 1; above 2^24 also a0 and a1 by one)
    const float slack = __fmul_rn(fabsf(rho), LONGK ? 0x1p-14f : 0x1p-15f);
    long long Zb = Z[0];
    float izb = iz[0];
#pragma unroll
    for (int b = 1; b < NB; b++)
        if (qb == b) {
            Zb = Z[b];
            izb = iz[b];
        }
    uint32_t words[EPG / 4];
#pragma unroll
    for (int w = 0; w < EPG / 4; w++) words[w] = 0;
#pragma unroll
    for (int j = 0; j < NT; j++) {
        const float v1 = __shfl_xor_sync(0xFFFFFFFFu, g < 4 ? acc[j][1] : acc[j][0], 16);
        const float v2 = __shfl_xor_sync(0xFFFFFFFFu, acc[j][3], 16);
        const float a0 = g < 4 ? acc[j][0] : v1, a1 = g < 4 ? v1 : acc[j][1], a2 = g < 4 ? acc[j][2] : v2;
        const float f0 = LONGK ? __int2float_rn(__float_as_int(a0)) : a0, f1 = LONGK ? __int2float_rn(__float_as_int(a1)) : a1,
                    f2 = LONGK ? __int2float_rn(__float_as_int(a2)) : a2;
        const float fn = __fmaf_rn(f2, 65536.0f, __fmaf_rn(f1, 256.0f, f0));
        const float c = q8_context(fn, izb, rho, slack, [&]() {
            auto i = [](float f) { return (long long)(LONGK ? __float_as_int(f) : __float2int_rn(f)); };
            return att_ctx_exact(i(a0) + i(a1) * 256 + i(a2) * 65536, Zb, rho);
        });
        words[j >> 2] |= (__float_as_uint(__fadd_rn(c, 12582912.0f)) & 0xFFu) << (8 * (j & 3));
    }
    if (qb < nb) store(qb, EPG * (2 * t + (g >= 4 ? 1 : 0)), words);  // rows past nb: none
}

}  // namespace mnmt
