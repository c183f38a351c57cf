// common.cuh -- device arithmetic shared by the sm_103a kernels of libmnmt.
//
// Every float operation here is written with explicit round-to-nearest
// intrinsics and the library is compiled with --fmad=false, so each a*b+c is
// two IEEE roundings exactly as the method's arithmetic is defined (the int8
// quantiser of App. B with zero point 0, the full-precision epilogues of Fig. 5,
// the fixed-point LayerNorm and softmax sums).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/mnmt.h"

#define MNMT_DEV __device__ __forceinline__

// ---------------------------------------------------------------------------
// programmatic dependent launch: every kernel of the library is launched
// allowed to start before its predecessor in the stream has finished; it lets
// its own successor launch at once, then waits for the predecessor (and the
// memory it wrote) before it reads anything.  Every kernel waits, so waiting
// for the predecessor also covers everything before it.
// ---------------------------------------------------------------------------
MNMT_DEV void pdl_allow_next() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
MNMT_DEV void pdl_grid_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// ---------------------------------------------------------------------------
// quantiser: q8(x, inv) = clamp(round_half_even(fl(x * inv)), -127, 127)
// ---------------------------------------------------------------------------
MNMT_DEV int8_t q8(float x, float inv) {
    float t = rintf(__fmul_rn(x, inv));
    t = fminf(fmaxf(t, -127.0f), 127.0f);
    return (int8_t)__float2int_rz(t);
}

// the same code as the low byte of a word: the clamp first (rne is monotone and
// +-127 are integers; a NaN becomes -127 either way), then rne by adding
// 1.5 2^23, whose low bits are the two's complement (conversion instructions
// run at an eighth of an addition's rate on this part)
MNMT_DEV uint32_t q8_bits(float x, float inv) {
    const float t = fminf(fmaxf(__fmul_rn(x, inv), -127.0f), 127.0f);
    return __float_as_uint(__fadd_rn(t, 12582912.0f));
}

// dequantise + bias: y = fl(fl(acc * fl(s_x * s_w)) + b)
MNMT_DEV float dequant_bias(int32_t acc, float s_x, float s_w, float b) {
    float sc = __fmul_rn(s_x, s_w);
    return __fadd_rn(__fmul_rn(__int2float_rn(acc), sc), b);
}

// ---------------------------------------------------------------------------
// round_half_even(v * 2^shift) as int64, with integer operations only.  Equal
// to llrint(ldexp((double)v, shift)) whenever |v| 2^shift < 2^62.
// ---------------------------------------------------------------------------
MNMT_DEV long long fx_scale(float v, int shift) {
    uint32_t bits = __float_as_uint(v);
    uint32_t ex = (bits >> 23) & 0xFFu;
    // fast path: v normal and y = v 2^shift a normal float below 2^62 -- the
    // scaling is then exact.  |y| >= 2^23 is an integer, its significand
    // shifted left; |y| < 2^23 rounds half to even into 32 bits (the 64-bit
    // float-to-integer conversion runs at a small fraction of this rate)
    if (ex != 0 && (int)ex + shift >= 1 && (int)ex + shift <= 127 + 61) {
        const int ey = (int)ex + shift;  // biased exponent of y
        if (ey >= 127 + 23) {
            const long long q = (long long)((bits & 0x7FFFFFu) | 0x800000u) << (ey - 150);
            return (bits >> 31) ? -q : q;
        }
        return (long long)__float2int_rn(__uint_as_float(bits + ((uint32_t)shift << 23)));
    }
    uint32_t man = bits & 0x7FFFFFu;
    int e;
    if (ex == 0) {
        e = -126 - 23;  // subnormal: value = man * 2^-149
    } else {
        man |= 0x800000u;
        e = (int)ex - 127 - 23;  // value = man * 2^e
    }
    int s = e + shift;
    long long q;
    if (s >= 0) {
        q = (long long)man << s;
    } else if (s < -25) {
        q = 0;  // man < 2^24: the value is below 1/2
    } else {
        int r = -s;
        uint32_t qq = man >> r;
        uint32_t rem = man & ((1u << r) - 1u);
        uint32_t half = 1u << (r - 1);
        if (rem > half || (rem == half && (qq & 1u))) qq++;
        q = (long long)qq;
    }
    return (bits >> 31) ? -q : q;
}

// exponent e with 2^(e-1) <= |v| < 2^e (0 for v == 0), as frexpf, read from the
// bits: normal v of biased exponent E gives E - 126; a subnormal with an
// n-bit significand gives n - 149
MNMT_DEV int exp_bound(float v) {
    const uint32_t a = __float_as_uint(v) & 0x7FFFFFFFu;
    const int E = (int)(a >> 23);
    if (E != 0) return E - 126;
    return a == 0 ? 0 : (32 - __clz((int)a)) - 149;
}

// ---------------------------------------------------------------------------
// e^x for x <= 0: Cody-Waite reduction with ln2 split into a 16-bit head and
// a tail, degree-7 Taylor polynomial of e^r by Horner in fused multiply-adds,
// scaled by 2^n through the exponent field; 0 below -87 and for a NaN.
// ---------------------------------------------------------------------------
MNMT_DEV float exp_own(float x) {
    if (!(x >= -87.0f)) return 0.0f;
    // n = rne(x log2(e)) in [-126, 0] by adding 1.5 2^23 (ulp 1 there: the sum
    // rounds the fraction half to even and its low bits hold n)
    const float t = __fadd_rn(__fmul_rn(x, 0x1.715476p+0f), 12582912.0f);
    const float n = __fsub_rn(t, 12582912.0f);
    float r = __fmaf_rn(-n, 0x1.62e4p-1f, x);
    r = __fmaf_rn(-n, 0x1.7f7d1cp-20f, r);
    float p = 0x1.a01a02p-13f;
    p = __fmaf_rn(p, r, 0x1.6c16c2p-10f);
    p = __fmaf_rn(p, r, 0x1.111112p-7f);
    p = __fmaf_rn(p, r, 0x1.555556p-5f);
    p = __fmaf_rn(p, r, 0x1.555556p-3f);
    p = __fmaf_rn(p, r, 0.5f);
    p = __fmaf_rn(p, r, 1.0f);
    p = __fmaf_rn(p, r, 1.0f);
    const int ni = (int)(__float_as_uint(t) - 0x4B400000u);
    float two_n = __uint_as_float((uint32_t)(ni + 127) << 23);
    return __fmul_rn(p, two_n);
}

// softmax weight on the 2^-24 grid: rne(exp(x) * 2^24), x <= 0
// (the float-to-integer conversion runs at 17 lanes per clock and SM on this
// part, an addition at 130: below 2^23 the rounding is an addition of 2^23,
// whose ulp is 1; from 2^23 on the value is an integer, read off its bits)
MNMT_DEV int32_t softmax_weight(float x) {
    const float w = __fmul_rn(exp_own(x), 16777216.0f);
    return w < 0x1p23f ? (int32_t)(__float_as_uint(__fadd_rn(w, 0x1p23f)) - 0x4B000000u)
                       : (int32_t)(__float_as_uint(w) - 0x4A800000u);
}

// natural log in double for z >= 1: z = f 2^k, f in [sqrt(1/2), sqrt(2)),
// ln f = 2 atanh(s), s = (f - 1)/(f + 1), odd series up to s^23.
MNMT_DEV double log_own(double z) {
    int k;
    double f = frexp(z, &k);
    if (f < 0x1.6a09e667f3bcdp-1) {
        f = __dmul_rn(f, 2.0);
        k = k - 1;
    }
    double s = __ddiv_rn(__dadd_rn(f, -1.0), __dadd_rn(f, 1.0));
    double s2 = __dmul_rn(s, s);
    double q = 0x1.642c8590b2164p-5;
    q = __dadd_rn(__dmul_rn(q, s2), 0x1.8618618618618p-5);
    q = __dadd_rn(__dmul_rn(q, s2), 0x1.af286bca1af28p-5);
    q = __dadd_rn(__dmul_rn(q, s2), 0x1.e1e1e1e1e1e1ep-5);
    q = __dadd_rn(__dmul_rn(q, s2), 0x1.1111111111111p-4);
    q = __dadd_rn(__dmul_rn(q, s2), 0x1.3b13b13b13b14p-4);
    q = __dadd_rn(__dmul_rn(q, s2), 0x1.745d1745d1746p-4);
    q = __dadd_rn(__dmul_rn(q, s2), 0x1.c71c71c71c71cp-4);
    q = __dadd_rn(__dmul_rn(q, s2), 0x1.2492492492492p-3);
    q = __dadd_rn(__dmul_rn(q, s2), 0x1.999999999999ap-3);
    q = __dadd_rn(__dmul_rn(q, s2), 0x1.5555555555555p-2);
    q = __dadd_rn(__dmul_rn(q, s2), 1.0);
    return __dadd_rn(__dmul_rn(__dmul_rn(2.0, s), q), __dmul_rn((double)k, 0x1.62e42fefa39efp-1));
}

// ---------------------------------------------------------------------------
// Ordering keys: a float and an index packed so that unsigned max picks the
// larger float, and between equal floats the lower index (-0 counts as +0).
// ---------------------------------------------------------------------------
MNMT_DEV uint32_t ordered_bits(float f) {
    uint32_t u = __float_as_uint(__fadd_rn(f, 0.0f));  // -0 + 0 = +0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
MNMT_DEV float from_ordered_bits(uint32_t o) {
    uint32_t u = (o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o;
    return __uint_as_float(u);
}
MNMT_DEV unsigned long long pack_key(float f, uint32_t idx) {
    return ((unsigned long long)ordered_bits(f) << 32) | (unsigned long long)(0xFFFFFFFFu - idx);
}
MNMT_DEV uint32_t key_index(unsigned long long k) { return 0xFFFFFFFFu - (uint32_t)(k & 0xFFFFFFFFull); }
MNMT_DEV float key_value(unsigned long long k) { return from_ordered_bits((uint32_t)(k >> 32)); }

// ---------------------------------------------------------------------------
// warp reductions
// ---------------------------------------------------------------------------
MNMT_DEV float warp_max_f(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}
MNMT_DEV long long warp_sum_ll(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}
MNMT_DEV int warp_sum_i(int v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}
MNMT_DEV unsigned long long warp_max_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long w = __shfl_xor_sync(0xFFFFFFFFu, v, o);
        v = w > v ? w : v;
    }
    return v;
}

// dp4a over 16 bytes held as int4
MNMT_DEV int dot16(int4 a, int4 b, int acc) {
    acc = __dp4a(a.x, b.x, acc);
    acc = __dp4a(a.y, b.y, acc);
    acc = __dp4a(a.z, b.z, acc);
    acc = __dp4a(a.w, b.w, acc);
    return acc;
}

// ---------------------------------------------------------------------------
// int8 codes as fp16 (exact) and back without conversion instructions: for an
// unsigned byte u, 0x6400 | u is the fp16 1024 + u; the code v = u - 128 has
// u = v ^ 0x80.  The fp16 1536 + v has v's two's complement as its low byte.
// ---------------------------------------------------------------------------
MNMT_DEV uint32_t h2_sub(uint32_t x, uint32_t y) {
    const __half2 r = __hsub2(*reinterpret_cast<const __half2 *>(&x), *reinterpret_cast<const __half2 *>(&y));
    return *reinterpret_cast<const uint32_t *>(&r);
}
MNMT_DEV uint32_t half2_sub_1024(uint32_t x) { return h2_sub(x, 0x64006400u); }
// four codes (bytes of w, lowest first) -> (v0, v1), (v2, v3)
MNMT_DEV void codes_to_half2(int w, uint32_t &lo, uint32_t &hi) {
    const uint32_t u = (uint32_t)w ^ 0x80808080u;
    lo = h2_sub(__byte_perm(u, 0x64646464u, 0x4140), 0x64806480u);  // 1152 = 1024 + 128
    hi = h2_sub(__byte_perm(u, 0x64646464u, 0x4342), 0x64806480u);
}
// (v0, v1), (v2, v3) -> four codes
MNMT_DEV uint32_t half2_to_codes(uint32_t lo, uint32_t hi) {
    return __byte_perm(h2_sub(lo, 0xE600E600u), h2_sub(hi, 0xE600E600u), 0x6420);  // v + 1536
}

// d += a b: m16n8k16, fp16 operands, fp32 accumulation
MNMT_DEV void mma_f16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ---------------------------------------------------------------------------
// Exact roundings to fp32 with integer operations only (no double precision,
// which is slow on this part).
// ---------------------------------------------------------------------------
// the float nearest S (ties to even), as __ll2float_rn, which runs at 2 lanes
// per clock and SM on this part: the top 32 significant bits, with the rest
// folded into the lowest one, round to 24 as the whole would
MNMT_DEV float ll2float(long long S) {
    const unsigned long long a = S < 0 ? 0ull - (unsigned long long)S : (unsigned long long)S;
    const int sh = __clzll((long long)(a | 1ull));
    const unsigned long long t = a << sh;
    const float f = __uint2float_rn((uint32_t)(t >> 32) | ((uint32_t)t ? 1u : 0u));
    const uint32_t b = __float_as_uint(f) + ((uint32_t)(32 - sh) << 23);
    return a == 0ull ? 0.0f : __uint_as_float(b | (S < 0 ? 0x80000000u : 0u));
}

// nearest float (ties to even) to S * 2^e, subnormals included
MNMT_DEV float rn32_pow2(long long S, int e) {
    if (S == 0) return 0.0f;
    {
        // fast path: the integer rounds to float once (half to even); scaling
        // by 2^e is exact while the result stays a normal float
        const float f = ll2float(S);
        const uint32_t fb = __float_as_uint(f);
        const int fe = (int)((fb >> 23) & 0xFFu) + e;
        if (fe >= 1 && fe <= 254) return __uint_as_float(fb + ((uint32_t)e << 23));
    }
    const unsigned long long a = S < 0 ? 0ull - (unsigned long long)S : (unsigned long long)S;
    const int nb = 64 - __clzll(a);  // significant bits of a
    const int E = nb - 1 + e;        // floor(log2 |value|)
    const int p = E >= -126 ? 24 : 150 + E;  // bits the float keeps
    const int shift = nb - p;
    unsigned long long q;
    if (shift <= 0) {
        q = a << (-shift);
    } else if (shift > 64) {
        q = 0;
    } else {
        q = shift == 64 ? 0ull : (a >> shift);
        const unsigned long long rem = shift == 64 ? a : (a & ((1ull << shift) - 1ull));
        const unsigned long long half = 1ull << (shift - 1);
        if (rem > half || (rem == half && (q & 1ull))) q++;
    }
    uint32_t bits;
    if (E >= -126) {
        int EE = E;
        if (q == (1ull << 24)) {
            q >>= 1;
            EE++;
        }
        bits = EE > 127 ? 0x7F800000u : (((uint32_t)(EE + 127) << 23) | (uint32_t)(q - (1ull << 23)));
    } else {
        bits = (uint32_t)q;  // subnormal, or the smallest normal after a carry
    }
    if (S < 0) bits |= 0x80000000u;
    return __uint_as_float(bits);
}

// nearest float (ties to even) to S * 2^e / d for 1 <= d <= 2048 and
// |S| < 2^63: the LayerNorm's mean and variance, S an exact fixed-point sum of
// d terms.  With d = z 2^k (z odd) and z = 1 this is rn32_pow2.  Otherwise
// |S| is shifted so the integer quotient q = floor(|S| 2^t / z) keeps at least
// 50 significant bits; the float keeps at most 24 of them, so the remainder
// only decides whether the value lies exactly on q or strictly above it, which
// one appended sticky bit (2q + [r != 0]) tells rn32_pow2 without moving the
// value across a rounding boundary.
MNMT_DEV float rn32_scaled_div(long long S, int e, int d) {
    const int k = __ffs(d) - 1;
    const unsigned z = (unsigned)d >> k;
    if (z == 1u) return rn32_pow2(S, e - k);
    if (S == 0) return 0.0f;
    const unsigned long long a = S < 0 ? 0ull - (unsigned long long)S : (unsigned long long)S;
    const int nb = 64 - __clzll(a);
    const int t = nb < 62 ? 62 - nb : 0;
    const unsigned long long num = a << t;
    const unsigned long long q = num / z, r = num - q * z;
    const float f = rn32_pow2((long long)(2ull * q + (r != 0ull ? 1ull : 0ull)), e - k - t - 1);
    return S < 0 ? -f : f;
}

// rn32_scaled_div for |S| < 2^63 with its 64-bit division replaced by a
// multiply-high by zm = floor(2^64 / z) (host-computed; d = z 2^kd, z odd): for
// a numerator below 2^63 the estimate is the quotient or one less, which the
// remainder corrects
MNMT_DEV float rn32_scaled_mul(long long S, int e, int kd, unsigned z, unsigned long long zm) {
    if (z == 1u) return rn32_pow2(S, e - kd);
    if (S == 0) return 0.0f;
    const unsigned long long a = S < 0 ? 0ull - (unsigned long long)S : (unsigned long long)S;
    const int nb = 64 - __clzll(a);
    const int t = nb < 62 ? 62 - nb : 0;
    const unsigned long long num = a << t;
    unsigned long long q = __umul64hi(num, zm), r = num - q * z;
    if (r >= z) {
        q++;
        r -= z;
    }
    const float f = rn32_pow2((long long)(2ull * q + (r != 0ull ? 1ull : 0ull)), e - kd - t - 1);
    return S < 0 ? -f : f;
}

// sign of a - X * 2^E for a < 2^62, X < 2^63
MNMT_DEV int cmp_scaled(unsigned long long a, unsigned long long X, int E) {
    if (E >= 0) {
        if (X == 0) return a > 0 ? 1 : 0;
        if (64 - __clzll(X) + E > 62) return -1;  // X 2^E >= 2^62 > a
        const unsigned long long v = X << E;
        return a > v ? 1 : (a < v ? -1 : 0);
    }
    const int s = -E;
    const unsigned long long qx = s >= 64 ? 0ull : (X >> s);
    const unsigned long long rx = s >= 64 ? X : (X & ((1ull << s) - 1ull));
    if (a > qx) return 1;
    if (a < qx) return -1;
    return rx ? -1 : 0;
}

// nearest float (ties to even) to the exact quotient n / z, |n| < 2^41, 1 <= z < 2^35
MNMT_DEV float rn32_div(long long n, long long z) {
    if (n == 0) return 0.0f;
    const unsigned long long a = n < 0 ? 0ull - (unsigned long long)n : (unsigned long long)n;
    float q = __fdiv_rn(__ull2float_rn(a), __ll2float_rn(z));  // within a few ulp of a / z
    for (int it = 0; it < 8; it++) {
        const uint32_t qb = __float_as_uint(q);
        const unsigned long long mq = (qb & 0x7FFFFFu) | 0x800000u;  // q = mq 2^eq (normal: a/z > 2^-35)
        const int eq = (int)((qb >> 23) & 0xFFu) - 150;
        // midpoint above: (2 mq + 1) 2^(eq-1); below: (2 mq - 1) 2^(eq-1), or (2^25 - 1) 2^(eq-2) at a power of two
        const int up = cmp_scaled(a, (unsigned long long)z * (2ull * mq + 1ull), eq - 1);
        if (up > 0 || (up == 0 && (mq & 1ull))) {
            q = __uint_as_float(qb + 1u);
            continue;
        }
        const bool pow2 = mq == 0x800000ull;
        const int dn = pow2 ? cmp_scaled(a, (unsigned long long)z * ((1ull << 25) - 1ull), eq - 2)
                            : cmp_scaled(a, (unsigned long long)z * (2ull * mq - 1ull), eq - 1);
        if (dn < 0 || (dn == 0 && (mq & 1ull))) {
            q = __uint_as_float(qb - 1u);
            continue;
        }
        break;
    }
    return n < 0 ? -q : q;
}

// fl(1 / fl(Z)) for q8_context.  Z >= 2^24 (the largest score's weight), or 0
// where no score is a number or the largest is infinite: every weight is then 0
// (a NaN difference has weight 0), N = 0, and the context is the code of 0.
MNMT_DEV float softmax_inv(float z) { return __frcp_rn(fmaxf(z, 1.0f)); }

// q8(nearest float to N / Z, rho), the quantised attention context of Eq. 2,
// from an approximation fN of N and invZ = softmax_inv(fl(Z)): t = fl(fl(fN invZ) rho) is off the exact chain by
// at most eight relative roundings of 2^-24 (two in fN, fl(Z), fl(1/Z), two
// products; the quotient and the product of the exact chain; < 2^-20) plus
// `slack`, what fN's absolute error makes of t.  Where t lies further from a
// rounding boundary than that (all but ~1e-4 of the values), rne(t) is the
// code; else exact() decides.  (A NaN clamps to -127, as in q8.)  Returns the
// code as an integer-valued float.
template <typename Exact>
MNMT_DEV float q8_context(float fN, float invZ, float rho, float slack, Exact exact) {
    const float t = fminf(fmaxf(__fmul_rn(__fmul_rn(fN, invZ), rho), -127.0f), 127.0f);
    const float r = __fsub_rn(__fadd_rn(t, 12582912.0f), 12582912.0f);  // rne for |t| < 2^22
    if (fabsf(__fsub_rn(t, r)) < __fsub_rn(0.5f, __fmaf_rn(fabsf(t), 0x1p-20f, slack))) return r;
    return exact();
}
// the same for N = 4096 hi + lo, |hi|, |lo| < 2^29 (up to 1024 keys): fl(lo) is
// off by at most 2^5, which makes at most rho 2^-19 of t
template <typename Exact>
MNMT_DEV int8_t q8_context_hl(int hi, int lo, float invZ, float rho, Exact exact) {
    const float fn = __fmaf_rn(__int2float_rn(hi), 4096.0f, __int2float_rn(lo));
    return (int8_t)(__float_as_uint(__fadd_rn(q8_context(fn, invZ, rho, __fmul_rn(fabsf(rho), 0x1p-18f), exact), 12582912.0f)) & 0xFFu);
}

// ---------------------------------------------------------------------------
// LayerNorm (App. A / App. D) of one row by one warp.  Mean and biased
// variance are exact fixed-point sums: the row's largest magnitude (an
// order-free maximum) sets a power-of-two grid on which every term is an
// integer below 2^52, summed in int64, so any reduction order gives the same
// bits; each sum / d is rounded once to fp32 (rn32_scaled_div); rstd =
// 1 / sqrt(var + 1e-5) in IEEE fp32; returns false if |x| >= 2^32.
// warp LayerNorm over a row held as VPL values per lane (element u*32 + lane, 0
// past d)
// ---------------------------------------------------------------------------
// exact warp sum of int64 values with |v| < 2^58 per lane: three 20-bit
// pieces summed by single-instruction warp reductions
MNMT_DEV long long warp_sum_exact(long long v) {
    int p0 = (int)(v & 0xFFFFF), p1 = (int)((v >> 20) & 0xFFFFF), p2 = (int)(v >> 40);
    p0 = __reduce_add_sync(0xFFFFFFFFu, p0);
    p1 = __reduce_add_sync(0xFFFFFFFFu, p1);
    p2 = __reduce_add_sync(0xFFFFFFFFu, p2);
    return (long long)p0 + (long long)p1 * (1LL << 20) + (long long)p2 * (1LL << 40);
}

// sum over v[0..N) of fx_scale(v[i], 52 - e) for |v[i]| <= 2^e, -70 <= e <= 33,
// without conversions or 64-bit shifts per term: T = rne(v 2^(52-e)) is taken
// apart as A 2^30 + B 2^8 + C, A = rne(v 2^(22-e)), B and C the same of the
// remainder 22 and 8 bits down.  Each rounding is an addition of 1.5 2^23, whose
// sum's low bits are the integer; each remainder is exact (a multiple of v's
// ulp, shorter than v); and A 2^30 + B 2^8 is even, so rounding the last
// remainder rounds T.  |A| <= 2^22, so int32 sums hold 2^9 terms.
template <int N>
MNMT_DEV long long fx_sum(const float (&v)[N], int e) {
    auto p2 = [](int k) { return __uint_as_float((uint32_t)(127 + k) << 23); };
    const float s22 = p2(22 - e), s44 = p2(44 - e), s52 = p2(52 - e);
    const float u22 = p2(e - 22), u44 = p2(e - 44);
    uint32_t sa = 0, sb = 0, sc = 0;
#pragma unroll
    for (int i = 0; i < N; i++) {
        const float ta = __fmaf_rn(v[i], s22, 12582912.0f);
        const float r1 = __fmaf_rn(-__fsub_rn(ta, 12582912.0f), u22, v[i]);
        const float tb = __fmaf_rn(r1, s44, 12582912.0f);
        const float r2 = __fmaf_rn(-__fsub_rn(tb, 12582912.0f), u44, r1);
        const float tc = __fmaf_rn(r2, s52, 12582912.0f);
        sa += __float_as_uint(ta);
        sb += __float_as_uint(tb);
        sc += __float_as_uint(tc);
    }
    const uint32_t off = (uint32_t)N * 0x4B400000u;  // the bits of 1.5 2^23, N times
    return (long long)(int)(sa - off) * (1LL << 30) + (long long)(int)(sb - off) * 256 + (int)(sc - off);
}

template <int VPL>
MNMT_DEV bool warp_layernorm(const float (&x)[VPL], int d, const float *__restrict__ g,
                             const float *__restrict__ b, float (&out)[VPL], int lane) {
    unsigned amax_bits = 0;
#pragma unroll
    for (int u = 0; u < VPL; u++)
        if (u * 32 + lane < d) amax_bits = max(amax_bits, __float_as_uint(x[u]) & 0x7FFFFFFFu);
    const float amax = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, amax_bits));
    if (!(amax < 0x1p32f)) return false;
    const int ea = exp_bound(amax);
    long long s1 = 0;
    if (ea >= -70) {
        s1 = fx_sum<VPL>(x, ea);
    } else {
#pragma unroll
        for (int u = 0; u < VPL; u++) s1 += fx_scale(x[u], 52 - ea);
    }
    const float mu = rn32_scaled_div(warp_sum_exact(s1), ea - 52, d);
    float c[VPL];
    unsigned bmax_bits = 0;
#pragma unroll
    for (int u = 0; u < VPL; u++) {
        c[u] = u * 32 + lane < d ? __fsub_rn(x[u], mu) : 0.0f;
        bmax_bits = max(bmax_bits, __float_as_uint(c[u]) & 0x7FFFFFFFu);
    }
    const int eb = exp_bound(__uint_as_float(__reduce_max_sync(0xFFFFFFFFu, bmax_bits)));
    long long s2 = 0;
    if (eb >= -36) {
        float c2[VPL];
        const float su = __uint_as_float((uint32_t)(127 - eb) << 23);
#pragma unroll
        for (int u = 0; u < VPL; u++) {
            const float cs = __fmul_rn(c[u], su);
            c2[u] = __fmul_rn(cs, cs);
        }
        s2 = fx_sum<VPL>(c2, 0);
    } else {
#pragma unroll
        for (int u = 0; u < VPL; u++) s2 += fx_scale(__fmul_rn(c[u], c[u]), 52 - 2 * eb);
    }
    s2 = warp_sum_exact(s2);
    const float var = rn32_scaled_div(s2, 2 * eb - 52, d);
    const float rstd = __fdiv_rn(1.0f, __fsqrt_rn(__fadd_rn(var, 1e-5f)));
#pragma unroll
    for (int u = 0; u < VPL; u++) {
        int i = u * 32 + lane;
        if (i < d) out[u] = __fadd_rn(__fmul_rn(__fmul_rn(c[u], rstd), g[i]), b[i]);
    }
    return true;
}

// device-side status word: first error wins
MNMT_DEV void set_status(int *status, int code) {
    if (status) atomicCAS(status, 0, code);
}
