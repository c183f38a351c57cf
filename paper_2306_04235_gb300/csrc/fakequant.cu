// fakequant.cu -- fake quantisation for quantisation-aware training (App. B
// "PTQ and QAT": the quantiser of Eq. quant inserted into the float model;
// besides the weights, its scale s is learnable).
//
//   symmetric, n bits: q = clamp(rne(fl(x fl(1/s))), -(2^(n-1)-1), 2^(n-1)-1), y = fl(q s)
//   min-max,   n bits: q = clamp(rne(fl(fl(x - r) fl(1/s))), 0, 2^n - 1),       y = fl(fl(q s) + r)
// Backward: straight-through for x, and the scale / offset gradients of the
// same expression with the rounding held fixed: with t the unrounded code and
// in = (qmin <= t <= qmax): dy/dx = in, dy/ds = in ? q - t : q, dy/dr = !in.
// The two scalar gradients are sums over the whole tensor, accumulated in
// fp64 precision (per-block partials combined with atomicAdd).
//
// The QAT forward of a linear quantises a float input per tensor (8-bit) and a
// float weight per row (learnable row scales), then runs the quantised linear
// of the codes -- the product X_q W_q^T is exact, so the result is that of the
// inference kernels on the same codes.
#include "common.cuh"
#include "internal.h"
#include "routes.h"

namespace mnmt {

struct FqRange {
    float qmin, qmax;
};

MNMT_DEV FqRange fq_range(int bits, int minmax) {
    if (minmax) return FqRange{0.0f, (float)((1 << bits) - 1)};
    const float m = (float)((1 << (bits - 1)) - 1);
    return FqRange{-m, m};
}

// the code of x as an integer-valued float: rne after the clamp (the bounds are
// integers and rne is monotone) by adding 1.5 2^23, with the sign of a zero as
// rne would leave it (rint and the conversions run at an eighth of an
// addition's rate on this part)
MNMT_DEV float fq_code(float x, float inv, float r, int minmax, FqRange rg, float *t_out) {
    const float t = minmax ? __fmul_rn(__fsub_rn(x, r), inv) : __fmul_rn(x, inv);
    if (t_out) *t_out = t;
    const float q = __fsub_rn(__fadd_rn(fminf(fmaxf(t, rg.qmin), rg.qmax), 12582912.0f), 12582912.0f);
    return minmax ? q : __uint_as_float(__float_as_uint(q) | (__float_as_uint(t) & 0x80000000u));
}
// an integer-valued |q| <= 255 as an int
MNMT_DEV int fq_int(float q) { return (int)(__float_as_uint(__fadd_rn(q, 12582912.0f)) - 0x4B400000u); }

__host__ __device__ __forceinline__ bool fq_al16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Forward, four elements per thread and step (groups; route_fake_quant) where
// every array is 16-byte aligned.  Bound by the 8 bytes per element (12 with
// codes) it moves.
template <bool GROUPS>
__global__ void fq_forward_kernel(const float *__restrict__ x, size_t n, float s, float r, int bits, int minmax,
                                  float *__restrict__ y, int32_t *__restrict__ codes) {
    const float inv = __fdiv_rn(1.0f, s);
    const FqRange rg = fq_range(bits, minmax);
    const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x, nt = (size_t)gridDim.x * blockDim.x;
    auto deq = [&](float q) {
        const float v = __fmul_rn(q, s);
        return minmax ? __fadd_rn(v, r) : v;
    };
    size_t done = 0;
    if (GROUPS) {
        for (size_t i = tid; i < n / 4; i += nt) {
            const float4 v = reinterpret_cast<const float4 *>(x)[i];
            const float q0 = fq_code(v.x, inv, r, minmax, rg, nullptr), q1 = fq_code(v.y, inv, r, minmax, rg, nullptr);
            const float q2 = fq_code(v.z, inv, r, minmax, rg, nullptr), q3 = fq_code(v.w, inv, r, minmax, rg, nullptr);
            if (codes) reinterpret_cast<int4 *>(codes)[i] = make_int4(fq_int(q0), fq_int(q1), fq_int(q2), fq_int(q3));
            if (y) reinterpret_cast<float4 *>(y)[i] = make_float4(deq(q0), deq(q1), deq(q2), deq(q3));
        }
        done = n & ~(size_t)3;
    }
    for (size_t i = done + tid; i < n; i += nt) {
        const float q = fq_code(x[i], inv, r, minmax, rg, nullptr);
        if (codes) codes[i] = fq_int(q);
        if (y) y[i] = deq(q);
    }
}

// s + e = a + b exactly (s = fl(a + b); no overflow)
MNMT_DEV float fq_two_sum(float a, float b, float &e) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

// Backward.  The scale gradient's terms g (q - t) are summed in fp64, whose
// pipe runs at 2 lanes per clock and SM on this part (six operations per
// element bounded the kernel: 31 us for 2 M elements): eight terms at a time
// are therefore first summed in fp32 pairs without loss.  q - t is exact in
// fp32 (|q - t| <= 1/2 and q = 0 or |t| >= 1/2); each product splits exactly
// into fl(p) and a remainder; two-sums carry every rounding error down twice,
// and the third level is added plainly (2^-72 of the largest term, far below
// fp64's own 2^-53).  Groups whose products leave the range in which that
// holds (2^-80 .. 2^120) are summed in fp64 term by term.  2 M elements: 14.8 us.
template <bool GROUPS>
__global__ void __launch_bounds__(256) fq_backward_kernel(const float *__restrict__ x, const float *__restrict__ g, size_t n, float s,
                                   float r, int bits, int minmax, float *__restrict__ gx, double *gs, double *gr) {
    const float inv = __fdiv_rn(1.0f, s);
    const FqRange rg = fq_range(bits, minmax);
    double as = 0.0, ar = 0.0;
    const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x, nt = (size_t)gridDim.x * blockDim.x;
    size_t done = 0;
    if (GROUPS) {
        for (size_t i = tid; i < n / 8; i += nt) {
            float xv[8], gv[8], ev[8], ov[8];
            *reinterpret_cast<float4 *>(xv) = reinterpret_cast<const float4 *>(x)[2 * i];
            *reinterpret_cast<float4 *>(xv + 4) = reinterpret_cast<const float4 *>(x)[2 * i + 1];
            *reinterpret_cast<float4 *>(gv) = reinterpret_cast<const float4 *>(g)[2 * i];
            *reinterpret_cast<float4 *>(gv + 4) = reinterpret_cast<const float4 *>(g)[2 * i + 1];
            float big = 0.0f, any = 0.0f;
            bool out = false;
#pragma unroll
            for (int k = 0; k < 8; k++) {
                float t;
                const float q = fq_code(xv[k], inv, r, minmax, rg, &t);
                const bool in = t >= rg.qmin && t <= rg.qmax;
                ov[k] = in ? gv[k] : 0.0f;
                ev[k] = in ? __fsub_rn(q, t) : q;
                out |= !in;
                big = fmaxf(big, fabsf(__fmul_rn(gv[k], ev[k])));
                any = fmaxf(any, fabsf(gv[k]));
                if (!(fabsf(gv[k]) <= 0x1p126f)) big = INFINITY;  // also a NaN, which fmaxf drops
            }
            reinterpret_cast<float4 *>(gx)[2 * i] = make_float4(ov[0], ov[1], ov[2], ov[3]);
            reinterpret_cast<float4 *>(gx)[2 * i + 1] = make_float4(ov[4], ov[5], ov[6], ov[7]);
            if (big >= 0x1p-80f && big <= 0x1p120f) {
                float sum = 0.0f, mid = 0.0f, low = 0.0f;
#pragma unroll
                for (int k = 0; k < 8; k++) {
                    const float p = __fmul_rn(gv[k], ev[k]), l = __fmaf_rn(gv[k], ev[k], -p);
                    float e1, e2;
                    sum = fq_two_sum(sum, p, e1);
                    mid = fq_two_sum(mid, l, e2);
                    low = __fadd_rn(low, e2);
                    mid = fq_two_sum(mid, e1, e2);
                    low = __fadd_rn(low, e2);
                }
                as += (double)sum;
                as += (double)mid;
                as += (double)low;
            } else if (any != 0.0f || big != 0.0f) {
#pragma unroll 1
                for (int k = 0; k < 8; k++) as += (double)gv[k] * (double)ev[k];
            }
            if (minmax && out) {
#pragma unroll
                for (int k = 0; k < 8; k++)
                    if (__float_as_uint(ov[k]) != __float_as_uint(gv[k])) ar += (double)gv[k];
            }
        }
        done = n & ~(size_t)7;
    }
    for (size_t i = done + tid; i < n; i += nt) {
        float t;
        const float q = fq_code(x[i], inv, r, minmax, rg, &t);
        const bool in = t >= rg.qmin && t <= rg.qmax;
        const float gi = g[i];
        gx[i] = in ? gi : 0.0f;
        as += (double)gi * (in ? (double)q - (double)t : (double)q);
        if (!in) ar += (double)gi;
    }
    // block reduction in fp64, then one atomic per block
    __shared__ double red_s[32], red_r[32];
    for (int o = 16; o > 0; o >>= 1) {
        as += __shfl_xor_sync(0xFFFFFFFFu, as, o);
        if (minmax) ar += __shfl_xor_sync(0xFFFFFFFFu, ar, o);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        red_s[warp] = as;
        red_r[warp] = ar;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double ts = 0.0, tr = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
            ts += red_s[w];
            tr += red_r[w];
        }
        atomicAdd(gs, ts);
        if (gr && minmax) atomicAdd(gr, tr);
    }
}

// The codes of a QAT linear in one launch: blocks [0, bx) quantise X [nx] per
// tensor, the others the rows of W [N][K] (K a multiple of 16) at their own
// scales, a warp per row; four elements per thread and step (16 bytes in, 4
// out) where the float arrays are 16-byte aligned.
__global__ void __launch_bounds__(256) fq_linear_codes_kernel(const float *__restrict__ X, size_t nx, float s_x, int bx,
                                                              const float *__restrict__ W, int N, int K,
                                                              const float *__restrict__ s_w, int bits,
                                                              int8_t *__restrict__ qx, int8_t *__restrict__ qw) {
    auto row = [](const float *src, int8_t *dst, size_t n, float inv, FqRange rg, size_t i0, size_t step) {
        if (fq_al16(src)) {
            for (size_t i = i0; i < n / 4; i += step) {
                const float4 v = reinterpret_cast<const float4 *>(src)[i];
                const uint32_t b0 = (uint32_t)fq_int(fq_code(v.x, inv, 0.0f, 0, rg, nullptr)),
                               b1 = (uint32_t)fq_int(fq_code(v.y, inv, 0.0f, 0, rg, nullptr)),
                               b2 = (uint32_t)fq_int(fq_code(v.z, inv, 0.0f, 0, rg, nullptr)),
                               b3 = (uint32_t)fq_int(fq_code(v.w, inv, 0.0f, 0, rg, nullptr));
                reinterpret_cast<uint32_t *>(dst)[i] =
                    __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
            }
        } else {
            for (size_t i = i0; i < n; i += step) dst[i] = (int8_t)fq_int(fq_code(src[i], inv, 0.0f, 0, rg, nullptr));
        }
    };
    if ((int)blockIdx.x < bx) {
        row(X, qx, nx, __fdiv_rn(1.0f, s_x), fq_range(8, 0), (size_t)blockIdx.x * 256 + threadIdx.x, (size_t)bx * 256);
        return;
    }
    const int nwarps = ((int)gridDim.x - bx) * 8;
    for (int n = ((int)blockIdx.x - bx) * 8 + (threadIdx.x >> 5); n < N; n += nwarps)
        row(W + (size_t)n * K, qw + (size_t)n * K, (size_t)K, __fdiv_rn(1.0f, s_w[n]), fq_range(bits, 0),
            (size_t)(threadIdx.x & 31), 32);
}

// blocks of 256 threads for n elements, `per` of them per thread and step
static int fq_grid(size_t n, int per) {
    size_t b = (n / per + 255) / 256;
    const size_t cap = (size_t)8 * device_sm_count();
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

cudaError_t launch_fake_quant(const float *x, size_t n, float s, float r, int bits, int minmax, float *y,
                              int32_t *codes, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const FqLaunch l = route_fake_quant(n, fq_al16(x) && fq_al16(y) && fq_al16(codes), false, minmax, device_sm_count());
    if (l.groups) fq_forward_kernel<true><<<l.blocks, 256, 0, st>>>(x, n, s, r, bits, minmax, y, codes);
    else fq_forward_kernel<false><<<l.blocks, 256, 0, st>>>(x, n, s, r, bits, minmax, y, codes);
    return cudaGetLastError();
}

cudaError_t launch_fake_quant_backward(const float *x, const float *g, size_t n, float s, float r, int bits,
                                       int minmax, float *gx, double *gs, double *gr, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(gs, 0, sizeof(double), st);
    if (e == cudaSuccess && gr) e = cudaMemsetAsync(gr, 0, sizeof(double), st);
    if (e != cudaSuccess || n == 0) return e;
    const FqLaunch l = route_fake_quant(n, fq_al16(x) && fq_al16(g) && fq_al16(gx), true, minmax, device_sm_count());
    if (l.groups) fq_backward_kernel<true><<<l.blocks, 256, 0, st>>>(x, g, n, s, r, bits, minmax, gx, gs, gr);
    else fq_backward_kernel<false><<<l.blocks, 256, 0, st>>>(x, g, n, s, r, bits, minmax, gx, gs, gr);
    return cudaGetLastError();
}

cudaError_t launch_fake_quant_linear(const float *X, const float *W, float s_x, const float *s_w, const float *bias,
                                     int M, int N, int K, int wbits, int8_t *qx, int8_t *qw, float *y,
                                     cudaStream_t st) {
    const size_t nx = (size_t)M * K;
    const int bx = fq_grid(nx, 4), bw = fq_grid((size_t)N * 32, 1);
    fq_linear_codes_kernel<<<bx + bw, 256, 0, st>>>(X, nx, s_x, bx, W, N, K, s_w, wbits, qx, qw);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    Epi e;
    memset(&e, 0, sizeof(e));
    e.mode = EPI_F32;
    e.s_x = s_x;
    e.s_w = s_w;
    e.bias = bias;
    e.f32 = y;
    e.ldf = N;
    return launch_linear(qx, K, qw, M, N, K, e, st);
}

}  // namespace mnmt
