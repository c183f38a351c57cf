// linear.cu -- quantised linear layers of the INT8 encoder-decoder (Sec. 3.3,
// Fig. 5; Eq. 3): int8 x int8 -> exact int32 accumulation, then a fused
// epilogue (dequantise with the per-channel weight scale, full-precision bias,
// then requantise / ReLU+requantise / gamma-residual / fp32 / K-V cache write /
// greedy argmax).
//
// Two kernels:
//   linear_smallm  M <= 16 rows, or up to 64 rows of a narrow layer, in chunks
//                  of <= 16 rows per grid row (batch-1 encoder, batch-1 and
//                  small-batch decode): every weight
//                  row is streamed once with 16-byte coalesced loads, the M
//                  activation rows sit in shared memory, products use dp4a and
//                  a lane group's partial sums meet by warp shuffles.  Bound by
//                  latency (start, loads, reduction).
//   linear_mma     other M > 16: CTA tiles of the int8 GEMM on the warp-level
//                  fp16 tensor-core instruction (mma.sync m16n8k16), the codes
//                  staged as bytes and widened to fp16 in registers; cp.async
//                  multi-stage pipeline with XOR-swizzled shared memory and
//                  ldmatrix fragment loads.  sm_103a has no int8 form of
//                  tcgen05.mma, and its mma.sync s8 runs at a quarter of the f16
//                  rate (542 against 2048 operations per clock and SM).
#include "common.cuh"
#include "epilogue.cuh"
#include "internal.h"

namespace mnmt {

// ---------------------------------------------------------------------------
// small-M path
// ---------------------------------------------------------------------------
constexpr int SM_THREADS = 256;
constexpr int SMALL_CHUNKED_MAX_M = 64;

// MT: rows held (>= M); LPC: lanes per weight row (K/16 chunks spread over
// LPC lanes); U: weight rows in flight per lane group.
// Bound by latency at these sizes.  The first weights are read before the rows
// of A are staged, and the lanes of a group share the reduction and the
// epilogue (gemv_reduce; one lane per group finishing all of a column's rows
// took as long as the products).  8 x 2048 x 512: 5.3 -> 2.8 us; 16 x 1536 x
// 512: 8.2 -> 3.6; 1 x 32000 x 256 argmax: 5.2 -> 4.4.
template <int MT, int LPC, int U>
__global__ void __launch_bounds__(SM_THREADS) linear_smallm(const int8_t *__restrict__ A, int lda,
                                                           const int8_t *__restrict__ W, int M, int N,
                                                           int K, Epi e) {
    pdl_grid_wait();
    if (e.skip && *e.skip) return;
    extern __shared__ int4 smA[];  // [MT][K/16]
    __shared__ unsigned long long s_best[MT];
    constexpr int NW = SM_THREADS / 32;
    constexpr int GPW = 32 / LPC;        // lane groups per warp
    constexpr int CPB = NW * GPW * U;    // columns per block pass
    constexpr int V = U * MT;
    const int kc = K >> 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = lane / LPC, sl = lane % LPC;
    // column of (warp, group, u): base + (u * NW + warp) * GPW + grp
    auto wload = [&](int base, int c, int4 (&w)[U]) {
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int n = base + (u * NW + warp) * GPW + grp;
            w[u] = (n < N && c < kc) ? __ldg(reinterpret_cast<const int4 *>(W + (size_t)n * K) + c) : make_int4(0, 0, 0, 0);
        }
    };
    int4 w[U];
    wload(blockIdx.x * CPB, sl, w);  // on its way while the rows of A are staged
    // blockIdx.y selects the chunk of MT rows this block computes
    const int m0 = blockIdx.y * MT;
    A += (size_t)m0 * lda;
    M -= m0;
    for (int i = threadIdx.x; i < MT * kc; i += SM_THREADS) {
        int m = i / kc, c = i - m * kc;
        smA[i] = (m < M) ? reinterpret_cast<const int4 *>(A + (size_t)m * lda)[c] : make_int4(0, 0, 0, 0);
    }
    if (threadIdx.x < MT) s_best[threadIdx.x] = 0ull;
    __syncthreads();
    const int t = e.t_ptr ? *e.t_ptr : 0;
    const bool argmax = e.mode == EPI_ARGMAX;
    constexpr int PER = V >= LPC ? V / LPC : 1;  // outputs a lane finishes per pass
    const int first = gemv_first<V, LPC>(sl);
    const bool owner = gemv_owner<V, LPC>(sl);
    unsigned long long best[PER];
#pragma unroll
    for (int i = 0; i < PER; i++) best[i] = 0ull;

    for (int base = blockIdx.x * CPB; base < N; base += gridDim.x * CPB) {
        int acc[V];
#pragma unroll
        for (int i = 0; i < V; i++) acc[i] = 0;
        for (int c0 = 0; c0 < kc; c0 += LPC) {
            const int c = c0 + sl;
            if (c0 || base != (int)blockIdx.x * CPB) wload(base, c, w);
            if (c < kc) {
#pragma unroll
                for (int m = 0; m < MT; m++) {
                    int4 a = smA[m * kc + c];
#pragma unroll
                    for (int u = 0; u < U; u++) acc[u * MT + m] = dot16(a, w[u], acc[u * MT + m]);
                }
            }
        }
        gemv_reduce<V, LPC>(acc, sl);
        // every residual load first: the stores may alias them
        float r[PER];
        if (e.mode == EPI_RESID) {
#pragma unroll
            for (int i = 0; i < PER; i++) {
                const int u = (first + i) / MT, m = (first + i) % MT, n = base + (u * NW + warp) * GPW + grp;
                r[i] = owner && n < N && m < M ? e.f32[(size_t)(m0 + m) * e.ldf + n] : 0.0f;
            }
        }
#pragma unroll
        for (int i = 0; i < PER; i++) {
            const int u = (first + i) / MT, m = (first + i) % MT, n = base + (u * NW + warp) * GPW + grp;
            if (!owner || n >= N || m >= M) continue;
            const float y = dequant_bias(acc[i], e.s_x, e.s_w[n], e.bias[n]);
            if (argmax) {
                const unsigned long long k = pack_key(y, (uint32_t)n);
                best[i] = k > best[i] ? k : best[i];
            } else if (e.mode == EPI_RESID) {
                e.f32[(size_t)(m0 + m) * e.ldf + n] = __fadd_rn(__fmul_rn(e.gamma, r[i]), y);
            } else {
                epi_store_y(e, m0 + m, n, y, t);
            }
        }
    }
    if (argmax) {
#pragma unroll
        for (int i = 0; i < PER; i++)
            if (best[i]) atomicMax(&s_best[(first + i) % MT], best[i]);
        __syncthreads();
        if (threadIdx.x < MT && (int)threadIdx.x < M) atomicMax(e.keys + m0 + threadIdx.x, s_best[threadIdx.x]);
    }
}

// ---------------------------------------------------------------------------
// tensor-core path (mma.sync f16 on the int8 codes)
// ---------------------------------------------------------------------------
MNMT_DEV uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

MNMT_DEV void cp_async16(uint32_t dst, const void *src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes));
}
MNMT_DEV void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
MNMT_DEV void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}
MNMT_DEV void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

// 64-byte shared rows, 16-byte chunks XOR-swizzled by (row / 2) % 4 so that the
// 8 rows of an ldmatrix phase hit 8 distinct bank groups.
MNMT_DEV int swz(int row, int chunk) { return row * 64 + ((chunk ^ ((row >> 1) & 3)) << 4); }

// An ldmatrix of bytes gives a lane four consecutive codes of one row per 16:
// widened to two fp16 pairs they are the two registers of an m16n8k16 fragment
// row, for a k order (codes 4 t .. 4 t + 3 of lane t) that A and W share.
// Products of codes are at most 2^14, so fp32 sums of 1024 of them are exact;
// BIGK (K > 1024) moves the sums to int32 every 1024.
// Bound by issue and the tensor pipe together (per warp and k-tile of a
// 128 x 128 block, 64 products of 8 cycles and ~340 issued instructions, 240 of
// them the widening).  Against the s8 instruction: 1000 x 1536 x 512 19.1 ->
// 9.1 us, 512 x 32000 x 512 argmax 158 -> 60 us, 8192 x 2048 x 512 180 -> 59 us.
template <int BM, int BN, int WARPS_M, int WARPS_N, int STAGES, bool BIGK>
__global__ void __launch_bounds__(WARPS_M *WARPS_N * 32)
    linear_mma(const int8_t *__restrict__ A, int lda, const int8_t *__restrict__ W, int M, int N, int K,
               Epi e) {
    constexpr int BK = 64;
    constexpr int NT = WARPS_M * WARPS_N * 32;
    constexpr int WTM = BM / WARPS_M, WTN = BN / WARPS_N;
    constexpr int MI = WTM / 16, NI = WTN / 8;
    static_assert(NI % 2 == 0, "B fragments are loaded two n8 tiles at a time");
    static_assert(STAGES * (BM + BN) * BK >= BM * (BN + 16), "the ring holds the int8 output tile");
    pdl_grid_wait();
    if (e.skip && *e.skip) return;
    extern __shared__ __align__(128) uint8_t smem[];
    uint8_t *sA = smem;
    uint8_t *sB = smem + STAGES * BM * BK;
    const int bm = blockIdx.y * BM, bn = blockIdx.x * BN;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = warp / WARPS_N, wn = warp % WARPS_N;
    const int ktiles = K / BK;

    float acc[MI][NI][4];
    int acci[BIGK ? MI : 1][BIGK ? NI : 1][4];
#pragma unroll
    for (int i = 0; i < MI; i++)
#pragma unroll
        for (int j = 0; j < NI; j++)
#pragma unroll
            for (int q = 0; q < 4; q++) {
                acc[i][j][q] = 0.0f;
                if (BIGK) acci[BIGK ? i : 0][BIGK ? j : 0][q] = 0;
            }

    auto load_stage = [&](int stage, int kt) {
        const int k0 = kt * BK;
        uint8_t *a_s = sA + stage * BM * BK;
        uint8_t *b_s = sB + stage * BN * BK;
#pragma unroll
        for (int i = threadIdx.x; i < BM * 4; i += NT) {
            int row = i >> 2, ch = i & 3;
            int g = bm + row;
            const int8_t *src = A + (size_t)(g < M ? g : M - 1) * lda + k0 + ch * 16;
            cp_async16(smem_u32(a_s + swz(row, ch)), src, g < M ? 16 : 0);
        }
#pragma unroll
        for (int i = threadIdx.x; i < BN * 4; i += NT) {
            int row = i >> 2, ch = i & 3;
            int g = bn + row;
            const int8_t *src = W + (size_t)(g < N ? g : N - 1) * K + k0 + ch * 16;
            cp_async16(smem_u32(b_s + swz(row, ch)), src, g < N ? 16 : 0);
        }
    };

#pragma unroll
    for (int s = 0; s < STAGES - 1; s++) {
        if (s < ktiles) load_stage(s, s);
        cp_async_commit();
    }
    for (int kt = 0; kt < ktiles; kt++) {
        cp_async_wait<STAGES - 2>();
        __syncthreads();
        {
            int nk = kt + STAGES - 1;
            if (nk < ktiles) load_stage(nk % STAGES, nk);
            cp_async_commit();
        }
        const uint8_t *a_s = sA + (kt % STAGES) * BM * BK;
        const uint8_t *b_s = sB + (kt % STAGES) * BN * BK;
#pragma unroll
        for (int kk = 0; kk < 2; kk++) {
            uint32_t ar[MI][4], br[NI / 2][4];
            const int j = lane >> 3, i8 = lane & 7;
#pragma unroll
            for (int mi = 0; mi < MI; mi++)
                ldmatrix_x4(ar[mi], smem_u32(a_s + swz(wm * WTM + mi * 16 + (j & 1) * 8 + i8, kk * 2 + (j >> 1))));
#pragma unroll
            for (int nj = 0; nj < NI / 2; nj++)
                ldmatrix_x4(br[nj], smem_u32(b_s + swz(wn * WTN + nj * 16 + (j >> 1) * 8 + i8, kk * 2 + (j & 1))));
#pragma unroll
            for (int h = 0; h < 2; h++) {  // the two k16 steps of these 32 codes
                uint32_t bf[NI][2];
#pragma unroll
                for (int ni = 0; ni < NI; ni++)
                    codes_to_half2((int)br[ni >> 1][2 * (ni & 1) + h], bf[ni][0], bf[ni][1]);
#pragma unroll
                for (int mi = 0; mi < MI; mi++) {
                    uint32_t af[4];
                    codes_to_half2((int)ar[mi][2 * h], af[0], af[2]);
                    codes_to_half2((int)ar[mi][2 * h + 1], af[1], af[3]);
#pragma unroll
                    for (int ni = 0; ni < NI; ni++) mma_f16_16816(acc[mi][ni], af, bf[ni][0], bf[ni][1]);
                }
            }
        }
        if (BIGK && ((kt & 15) == 15 || kt == ktiles - 1)) {
#pragma unroll
            for (int mi = 0; mi < MI; mi++)
#pragma unroll
                for (int ni = 0; ni < NI; ni++)
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        acci[BIGK ? mi : 0][BIGK ? ni : 0][q] += __float2int_rn(acc[mi][ni][q]);
                        acc[mi][ni][q] = 0.0f;
                    }
        }
    }
    cp_async_wait<0>();
    if (BIGK) {
#pragma unroll
        for (int mi = 0; mi < MI; mi++)
#pragma unroll
            for (int ni = 0; ni < NI; ni++)
#pragma unroll
                for (int q = 0; q < 4; q++) acc[mi][ni][q] = __int2float_rn(acci[BIGK ? mi : 0][BIGK ? ni : 0][q]);
    }

    // y in place: lane (g, tq) holds rows g, g + 8 and columns 2 tq, 2 tq + 1 of every 16 x 8 tile
    const int g = lane >> 2, tq = lane & 3;
    const int row0 = bm + wm * WTM + g, col0 = bn + wn * WTN + 2 * tq;
#pragma unroll
    for (int ni = 0; ni < NI; ni++) {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            const int col = col0 + ni * 8 + c;
            const float sc = col < N ? __fmul_rn(e.s_x, e.s_w[col]) : 0.0f, bs = col < N ? e.bias[col] : 0.0f;
#pragma unroll
            for (int mi = 0; mi < MI; mi++) {
                acc[mi][ni][c] = __fadd_rn(__fmul_rn(acc[mi][ni][c], sc), bs);
                acc[mi][ni][2 + c] = __fadd_rn(__fmul_rn(acc[mi][ni][2 + c], sc), bs);
            }
        }
    }
    if (e.mode == EPI_ARGMAX) {
        // per row: the largest (ordered y, lowest column) of this thread's
        // columns, the quad's, then the block's (one atomic per row and block)
        __syncthreads();
        unsigned long long *best_s = reinterpret_cast<unsigned long long *>(smem);  // [WARPS_N][BM]
#pragma unroll
        for (int mi = 0; mi < MI; mi++) {
#pragma unroll
            for (int hr = 0; hr < 2; hr++) {
                uint32_t bo = 0u, bc = 0u;
#pragma unroll
                for (int ni = 0; ni < NI; ni++) {
#pragma unroll
                    for (int c = 0; c < 2; c++) {
                        const uint32_t col = (uint32_t)(col0 + ni * 8 + c);
                        const uint32_t o = col < (uint32_t)N ? ordered_bits(acc[mi][ni][2 * hr + c]) : 0u;
                        if (o > bo) {
                            bo = o;
                            bc = col;
                        }
                    }
                }
                unsigned long long best = bo ? ((unsigned long long)bo << 32) | (0xFFFFFFFFu - bc) : 0ull;
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {
                    unsigned long long w2 = __shfl_xor_sync(0xFFFFFFFFu, best, o);
                    best = w2 > best ? w2 : best;
                }
                if (tq == 0) best_s[wn * BM + wm * WTM + mi * 16 + hr * 8 + g] = best;
            }
        }
        __syncthreads();
        for (int r = threadIdx.x; r < BM && bm + r < M; r += NT) {
            unsigned long long best = best_s[r];
#pragma unroll
            for (int w = 1; w < WARPS_N; w++) best = best_s[w * BM + r] > best ? best_s[w * BM + r] : best;
            atomicMax(e.keys + bm + r, best);
        }
        return;
    }
    if (e.mode == EPI_RESID || e.mode == EPI_F32) {
        // two adjacent columns per access where they are 8-byte aligned; every
        // residual load of an m-tile before its stores
        const bool v2 = e.ldf % 2 == 0 && (reinterpret_cast<uintptr_t>(e.f32) & 7) == 0;
#pragma unroll
        for (int mi = 0; mi < MI; mi++) {
            if (e.mode == EPI_RESID) {
                float r[NI][4];
#pragma unroll
                for (int ni = 0; ni < NI; ni++)
#pragma unroll
                    for (int hr = 0; hr < 2; hr++) {
                        const int row = row0 + mi * 16 + hr * 8, col = col0 + ni * 8;
                        const float *p = e.f32 + (size_t)row * e.ldf + col;
                        float2 v = make_float2(0.0f, 0.0f);
                        if (row < M && col + 1 < N && v2) v = *reinterpret_cast<const float2 *>(p);
                        else if (row < M) {
                            if (col < N) v.x = p[0];
                            if (col + 1 < N) v.y = p[1];
                        }
                        r[ni][2 * hr] = v.x;
                        r[ni][2 * hr + 1] = v.y;
                    }
#pragma unroll
                for (int ni = 0; ni < NI; ni++)
#pragma unroll
                    for (int q = 0; q < 4; q++)
                        acc[mi][ni][q] = __fadd_rn(__fmul_rn(e.gamma, r[ni][q]), acc[mi][ni][q]);
            }
#pragma unroll
            for (int ni = 0; ni < NI; ni++)
#pragma unroll
                for (int hr = 0; hr < 2; hr++) {
                    const int row = row0 + mi * 16 + hr * 8, col = col0 + ni * 8;
                    float *p = e.f32 + (size_t)row * e.ldf + col;
                    if (row < M && col + 1 < N && v2) {
                        *reinterpret_cast<float2 *>(p) = make_float2(acc[mi][ni][2 * hr], acc[mi][ni][2 * hr + 1]);
                    } else if (row < M) {
                        if (col < N) p[0] = acc[mi][ni][2 * hr];
                        if (col + 1 < N) p[1] = acc[mi][ni][2 * hr + 1];
                    }
                }
        }
        return;
    }
    const int t = e.t_ptr ? *e.t_ptr : 0;
    if ((e.mode == EPI_Q8 || e.mode == EPI_RELU_Q8) && !e.out16 && e.ldo % 16 == 0 &&
        (reinterpret_cast<uintptr_t>(e.out) & 15) == 0) {
        // int8 rows through shared memory (rows of BN + 16 bytes), 16 bytes per store
        constexpr int LDS = BN + 16;
        __syncthreads();
#pragma unroll
        for (int ni = 0; ni < NI; ni++) {
            const int col = col0 + ni * 8;
            const float i0 = col < N ? e.inv_out[col] : 0.0f, i1 = col + 1 < N ? e.inv_out[col + 1] : 0.0f;
#pragma unroll
            for (int mi = 0; mi < MI; mi++)
#pragma unroll
                for (int hr = 0; hr < 2; hr++) {
                    float y0 = acc[mi][ni][2 * hr], y1 = acc[mi][ni][2 * hr + 1];
                    if (e.mode == EPI_RELU_Q8) {
                        y0 = y0 > 0.0f ? y0 : 0.0f;
                        y1 = y1 > 0.0f ? y1 : 0.0f;
                    }
                    *reinterpret_cast<uint16_t *>(smem + (wm * WTM + mi * 16 + hr * 8 + g) * LDS + wn * WTN + ni * 8 + 2 * tq) =
                        (uint16_t)__byte_perm(q8_bits(y0, i0), q8_bits(y1, i1), 0x0040);
                }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < BM * (BN / 16); i += NT) {
            const int r = i / (BN / 16), c = (i % (BN / 16)) * 16, row = bm + r, col = bn + c;
            if (row >= M || col >= N) continue;
            const uint4 v = *reinterpret_cast<const uint4 *>(smem + r * LDS + c);
            if (col + 16 <= N) {
                *reinterpret_cast<uint4 *>(e.out + (size_t)row * e.ldo + col) = v;
            } else {
                for (int b = 0; col + b < N; b++) e.out[(size_t)row * e.ldo + col + b] = (int8_t)smem[r * LDS + c + b];
            }
        }
        return;
    }
#pragma unroll
    for (int mi = 0; mi < MI; mi++)
#pragma unroll
        for (int ni = 0; ni < NI; ni++)
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int row = row0 + mi * 16 + (q >> 1) * 8, col = col0 + ni * 8 + (q & 1);
                if (row < M && col < N) epi_store_y(e, row, col, acc[mi][ni][q], t);
            }
}

// ---------------------------------------------------------------------------
// dispatch
// ---------------------------------------------------------------------------
template <int BM, int BN, int WM, int WN, int STAGES>
static cudaError_t mma_attr() {
    cudaError_t err = cudaFuncSetAttribute(linear_mma<BM, BN, WM, WN, STAGES, false>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, STAGES * (BM + BN) * 64);
    if (err == cudaSuccess)
        err = cudaFuncSetAttribute(linear_mma<BM, BN, WM, WN, STAGES, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   STAGES * (BM + BN) * 64);
    return err;
}

// Opt the tensor-core kernels into their shared memory (once per process,
// before any launch or stream capture).
cudaError_t linear_init() {
    cudaError_t err = mma_attr<128, 128, 2, 4, 4>();
    if (err == cudaSuccess) err = mma_attr<64, 64, 2, 2, 4>();
    return err;
}

template <int MT, int LPC, int U>
static cudaError_t launch_small_u(const int8_t *A, int lda, const int8_t *W, int M, int N, int K, const Epi &e,
                                  cudaStream_t st) {
    constexpr int CPB = (SM_THREADS / 32) * (32 / LPC) * U;
    int blocks = (N + CPB - 1) / CPB;
    if (blocks > 4 * device_sm_count()) blocks = 4 * device_sm_count();
    const dim3 grid(blocks, (M + MT - 1) / MT);  // row chunks of MT, one per grid row
    launch_pdl(linear_smallm<MT, LPC, U>, grid, SM_THREADS, (size_t)MT * K, st, A, lda, W, M, N, K, e);
    return cudaGetLastError();
}

// two weight rows per lane group and pass, or one where that leaves fewer
// blocks than SMs
template <int MT, int LPC>
static cudaError_t launch_small_t(const int8_t *A, int lda, const int8_t *W, int M, int N, int K, const Epi &e,
                                  cudaStream_t st) {
    constexpr int CPB2 = (SM_THREADS / 32) * (32 / LPC) * 2;
    const long blocks = (long)((N + CPB2 - 1) / CPB2) * ((M + MT - 1) / MT);
    return blocks >= device_sm_count() ? launch_small_u<MT, LPC, 2>(A, lda, W, M, N, K, e, st)
                         : launch_small_u<MT, LPC, 1>(A, lda, W, M, N, K, e, st);
}

template <int MT>
static cudaError_t launch_small(const int8_t *A, int lda, const int8_t *W, int M, int N, int K, const Epi &e,
                                cudaStream_t st) {
    const int kc = K / 16;
    if ((size_t)MT * K > 48 * 1024) return cudaErrorInvalidValue;  // K <= 3072 at M <= 16
    if (kc >= 32) return launch_small_t<MT, 32>(A, lda, W, M, N, K, e, st);
    if (kc >= 16) return launch_small_t<MT, 16>(A, lda, W, M, N, K, e, st);
    return launch_small_t<MT, 8>(A, lda, W, M, N, K, e, st);
}

template <int BM, int BN, int WM, int WN, int STAGES>
static cudaError_t launch_mma(const int8_t *A, int lda, const int8_t *W, int M, int N, int K, const Epi &e,
                              cudaStream_t st) {
    auto k = K > 1024 ? linear_mma<BM, BN, WM, WN, STAGES, true> : linear_mma<BM, BN, WM, WN, STAGES, false>;
    size_t smem = (size_t)STAGES * (BM + BN) * 64;
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM);
    launch_pdl(k, grid, WM * WN * 32, smem, st, A, lda, W, M, N, K, e);
    return cudaGetLastError();
}

cudaError_t launch_linear(const int8_t *A, int lda, const int8_t *W, int M, int N, int K, const Epi &e,
                          cudaStream_t st) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    if (M <= 16) {
        if (M == 1) return launch_small<1>(A, lda, W, M, N, K, e, st);
        if (M <= 2) return launch_small<2>(A, lda, W, M, N, K, e, st);
        if (M <= 4) return launch_small<4>(A, lda, W, M, N, K, e, st);
        if (M <= 8) return launch_small<8>(A, lda, W, M, N, K, e, st);
        return launch_small<16>(A, lda, W, M, N, K, e, st);
    }
    // up to 64 rows over few output tiles (narrow N): chunks of 16 rows over
    // the grid's y dimension spread the work over more blocks than the 64 x 64
    // tiling would (the weights are re-read per chunk, from L2)
    const long tiles64 = (long)((M + 63) / 64) * ((N + 63) / 64);
    if (M <= SMALL_CHUNKED_MAX_M && K <= 2048 && tiles64 < 8) return launch_small<16>(A, lda, W, M, N, K, e, st);
    long tiles_big = (long)((M + 127) / 128) * ((N + 127) / 128);
    if (tiles_big >= device_sm_count()) return launch_mma<128, 128, 2, 4, 4>(A, lda, W, M, N, K, e, st);
    return launch_mma<64, 64, 2, 2, 4>(A, lda, W, M, N, K, e, st);
}

}  // namespace mnmt
