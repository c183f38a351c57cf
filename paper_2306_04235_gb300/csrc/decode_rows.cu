// decode_rows.cu -- one decoder step (all layers) of a batch of hypotheses on
// independent thread-block clusters.
//
// A batched decode step run as one kernel per operation is a chain of ~11
// launches per layer, each for well under a microsecond of work: at 512 rows
// the linears kept the tensor pipe 1-4 % busy.  The rows of a step depend on
// one another only in the beam selection that follows it, so here a cluster of
// H / HPC CTAs (HPC heads each) takes 8 NB rows (NB = 1, 2 or 4) through the
// whole decoder:
//   * a linear is split by output columns over the CTAs; Q, K and V of a head
//     land in one CTA, which attends over them without an exchange;
//   * products run on the warp-level tensor cores with the weights as the
//     16-row operand and the rows as its 8-column one (mma.sync m16n8k16 on
//     fp16 integers widened in registers from int8; fp32 sums of up to 1024
//     products are exact, K = 2048 adds two);
//   * the weights stream through a ring of 8 KB slots by bulk copies issued by
//     a producer warp that runs ahead over layer and phase boundaries; they are
//     laid out once per session in the order the warps consume them, as
//     operand fragments (dr_pack);
//   * the fp32 residual lives with the CTA that owns the row: the W_o / W_2
//     outputs go to the row's owner, which adds them, normalises and sends the
//     codes to every CTA; exchanges are st.async stores completing on the
//     receiver's mbarrier (two, alternating, armed by the receiver for the
//     phase after next).
// No cluster waits for another, so it would run in any number of waves; one is
// where it is faster (route_rows_variant).  The
// arithmetic is that of the other kernels (exact integer sums, the same fp32
// roundings), so results are bit-identical.
// Bound by the chain of short phases (time stamps of one step, 16 clusters of
// the 2-layer, d = 256 model: 63 us -- linears 1 to 2.6 us, attention 3 to 5,
// LayerNorm with its two exchanges 2.8 each): issue, instruction fetch and
// exchange latency, not memory or the tensor pipe.
#include <cstddef>
#include <type_traits>

#include "attn_core.cuh"
#include "common.cuh"
#include "decode_rows.h"
#include "epilogue.cuh"
#include "internal.h"
#include "mbarrier.cuh"

namespace mnmt {
namespace {

constexpr int DR_WARPS = 8;                         // compute warps
constexpr int DR_THREADS = DR_WARPS * 32 + 32;      // and the producer warp
constexpr int DR_SLOT = 8192;                       // ring slot: one 1 KB tile per compute warp
constexpr int DR_MAX_SLOTS = 16;

enum { DR_QKV = 0, DR_O = 1, DR_Q2 = 2, DR_O2 = 3, DR_W1 = 4, DR_W2 = 5 };
// exchanges of a step: the input codes of layer 0, then nine per layer (the
// last layer's final one does not happen)
enum { DX_A = 0, DX_CTX = 1, DX_Y = 2, DX_H = 3 };
__host__ __device__ constexpr int dr_exchange_kind(int x) {
    return x == 0 ? DX_A : ((x - 1) % 9 == 6 ? DX_H : ((x - 1) % 3 == 0 ? DX_CTX : ((x - 1) % 3 == 1 ? DX_Y : DX_A)));
}

// how a phase's output tiles (16 columns each) are spread over the warps: K in
// two halves when their number is 4 or 12 (each warp one or three tiles of a
// half), else whole (a warp every eighth tile); tpw = 0: unsupported
struct DrSplit {
    int ks2, tpw;
};
__host__ __device__ constexpr DrSplit dr_split(int tiles) {
    return tiles == 4 || tiles == 12 ? DrSplit{1, tiles / 4} : tiles % 8 == 0 && tiles <= 32 ? DrSplit{0, tiles / 8} : DrSplit{0, 0};
}
// columns of a phase per CTA
__host__ __device__ constexpr int dr_cols(int phase, int hpc, int F, int nc) {
    return phase == DR_QKV ? 192 * hpc : phase == DR_W1 ? F / nc : 64 * hpc;
}

// ---------------------------------------------------------------------------
// weight packing: slot by slot, warp w's 1 KB is the operand fragments of its
// tile and k-block: lane (g, t) = (lane / 4, lane % 4) holds the 16 codes
// [16 t, 16 t + 16) of the k-block of row g, then (512 bytes on) of row g + 8
// ---------------------------------------------------------------------------
__global__ void dr_pack_kernel(const __grid_constant__ DrPack pk, int d, int nc, int hpc, int F, uint8_t *__restrict__ out,
                               size_t cta_bytes) {
    const int layer = blockIdx.y / 6, phase = blockIdx.y % 6;
    size_t off = cta_bytes / pk.n_dec * layer;
    int cols = 0, K = 0;
    for (int p = 0; p <= phase; p++) {
        off += (size_t)cols * K;
        cols = dr_cols(p, hpc, F, nc);
        K = p == DR_W2 ? F : d;
    }
    const DrSplit sp = dr_split(cols / 16);
    const int per_cta = cols * K / 16;  // 16-byte pieces
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= per_cta * nc) return;
    const int c = i / per_cta, p = i - c * per_cta;
    const int lane = p & 31, half = (p >> 5) & 1, w = (p >> 6) & 7, slot = p >> 9;
    const int kb = slot / sp.tpw, ti = slot - kb * sp.tpw;
    const int kh = sp.ks2 ? (w & 1) : 0, wt = sp.ks2 ? (w >> 1) : w, nwt = sp.ks2 ? 4 : 8;
    const int nkb = (sp.ks2 ? K / 2 : K) / 64;
    const int nl = (wt + nwt * ti) * 16 + (lane >> 2) + 8 * half, hc = 64 * hpc;
    const int n = phase == DR_QKV ? nl / hc * d + hc * c + nl % hc : c * cols + nl;
    const int k = (kh * nkb + kb) * 64 + 16 * (lane & 3);
    reinterpret_cast<int4 *>(out + (size_t)c * cta_bytes + off)[p] =
        *reinterpret_cast<const int4 *>(pk.w[layer][phase] + (size_t)n * K + k);
}

// ---------------------------------------------------------------------------
// cluster helpers
// ---------------------------------------------------------------------------
MNMT_DEV uint32_t dr_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
MNMT_DEV uint32_t dr_mapa(uint32_t local, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
MNMT_DEV void dr_send4(uint32_t remote, uint4 v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];\n" ::"r"(
                     remote),
                 "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
                 : "memory");
}
MNMT_DEV void dr_send2(uint32_t remote, uint32_t x, uint32_t y, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];\n" ::"r"(remote),
                 "r"(x), "r"(y), "r"(bar)
                 : "memory");
}
// [p, p + bytes) to L2 (16-byte aligned)
MNMT_DEV void dr_prefetch(const void *p, int bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(p), "r"(bytes) : "memory");
}
// barrier over the compute warps
MNMT_DEV void dr_sync() { asm volatile("bar.sync 1, %0;" ::"n"(DR_WARPS * 32) : "memory"); }
// barrier over all warps
MNMT_DEV void dr_sync_all() { asm volatile("bar.sync 0, %0;" ::"n"(DR_THREADS) : "memory"); }

// state of a CTA's pipeline that every wait shares: once a wait has given up,
// the later ones return at once (the step's results are void: status is set)
// and the CTA leaves by dr_leave's longer way.  A thread whose wait for an
// exchange has given up sends nothing more and arms no exchange barrier (it has
// not seen the phase end); the peers that miss its bytes give up too.
struct DrWait {
    int *status;
    volatile uint32_t *abort_flag;
    MNMT_DEV bool operator()(uint32_t bar, uint32_t parity) const {
        if (mbar_test(bar, parity)) return true;
        if (*abort_flag) return false;
        if (mbar_wait(bar, parity)) return true;
        *abort_flag = 1;
        set_status(status, MNMT_ETIMEOUT);
        return false;
    }
};

// what the out-of-line pieces of the kernel need, from the parameter block at
// the start of shared memory.  (The kernel walks its code once per layer; pieces
// used more than once are single copies, as instruction fetch was the largest
// stall when everything was inlined.)
struct DrPipe {
    const uint8_t *ring;
    uint32_t full, empty, xbars;
    int slots;
    DrWait wait;
};
// the CTA's abort flag, behind the barriers
MNMT_DEV volatile uint32_t *dr_abort(const DrParams &P) {
    return reinterpret_cast<volatile uint32_t *>(const_cast<uint8_t *>(reinterpret_cast<const uint8_t *>(&P)) + P.off_bar +
                                                 8 * (2 * DR_MAX_SLOTS + 2));
}
MNMT_DEV DrPipe dr_pipe(const DrParams &P) {
    const uint8_t *sm = reinterpret_cast<const uint8_t *>(&P);
    const uint32_t bars = dr_smem(sm + P.off_bar);
    return DrPipe{sm + P.off_ring, bars, bars + 8u * DR_MAX_SLOTS, bars + 16u * DR_MAX_SLOTS, P.slots, DrWait{P.status, dr_abort(P)}};
}

// The way out of a CTA whose wait has timed out (every thread).  Other CTAs of
// the cluster may still send to it: it stays until all of them have ended or
// come here too (the cluster barrier counts ended threads as arrived, and every
// wait on the way is bounded), and then for as long again as a store needs to
// land many times over.  A CTA without a timed-out wait just ends: every byte
// that the others send it in a step has arrived by its last exchange.
constexpr unsigned long long DR_LAND_NS = 100000;
__device__ __noinline__ void dr_leave() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;\n" ::: "memory");
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < DR_LAND_NS) {
    }
}

// this warp's tiles of one linear over k-blocks [0, nkb): acc[i][nt] = W tile x
// rows; `it` counts the ring slots consumed so far.  The next tile's weights
// are read before this tile's products: a tile is a chain (barrier test, read,
// widening, four dependent products) that two warps per scheduler do not hide.
template <int NB, int TPW>
MNMT_DEV void dr_gemm(const int8_t *ap, int stride, int nkb, const uint8_t *ring, uint32_t full, uint32_t empty, int slots,
                      uint32_t &it, const DrWait &wait, float (&acc)[TPW][NB][4]) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < TPW; i++)
#pragma unroll
        for (int nt = 0; nt < NB; nt++)
#pragma unroll
            for (int q = 0; q < 4; q++) acc[i][nt][q] = 0.0f;
    uint32_t s = it % (uint32_t)slots, par = (it / (uint32_t)slots) & 1;
    const uint8_t *wp = ring + warp * 1024 + lane * 16;
    int4 w0, w1;
    auto fetch = [&]() {
        wait(full + 8u * s, par);
        const int4 *tp = reinterpret_cast<const int4 *>(wp + s * DR_SLOT);
        w0 = tp[0];
        w1 = tp[32];
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + 8u * s);
        if (++s == (uint32_t)slots) {
            s = 0;
            par ^= 1;
        }
    };
    fetch();
    for (int kb = 0; kb < nkb; kb++) {
        int4 av[NB];
#pragma unroll
        for (int nt = 0; nt < NB; nt++) av[nt] = *reinterpret_cast<const int4 *>(ap + nt * 8 * stride + kb * 64);
        uint32_t bf[NB][4][2];
#pragma unroll
        for (int nt = 0; nt < NB; nt++) {
            codes_to_half2(av[nt].x, bf[nt][0][0], bf[nt][0][1]);
            codes_to_half2(av[nt].y, bf[nt][1][0], bf[nt][1][1]);
            codes_to_half2(av[nt].z, bf[nt][2][0], bf[nt][2][1]);
            codes_to_half2(av[nt].w, bf[nt][3][0], bf[nt][3][1]);
        }
#pragma unroll
        for (int i = 0; i < TPW; i++) {
            const int u0[4] = {w0.x, w0.y, w0.z, w0.w}, u1[4] = {w1.x, w1.y, w1.z, w1.w};
            if (i + 1 < TPW || kb + 1 < nkb) fetch();
#pragma unroll
            for (int k = 0; k < 4; k++) {
                uint32_t a[4];
                codes_to_half2(u0[k], a[0], a[2]);
                codes_to_half2(u1[k], a[1], a[3]);
#pragma unroll
                for (int nt = 0; nt < NB; nt++) mma_f16_16816(acc[i][nt], a, bf[nt][k][0], bf[nt][k][1]);
            }
        }
    }
    it += (uint32_t)(nkb * TPW);
}

// One linear: the products, the halves of K joined through `red`, y = fl(fl(acc
// sc) + b); column n of the CTA is column base + n + n / HC * seg of the layer.
// Q8 = false: y as fp32 to dst [row][ldo]; else its (ReLU'd) code.
template <int NB, int HC, int TPW, bool KS2, bool Q8>
__device__ __noinline__ void dr_linear(const DrParams &P, const DrLin &L, int base, int seg, const int8_t *act, int stride,
                                       int K, uint32_t it, uint8_t *dst, int ldo, bool relu) {
    const DrPipe pp = dr_pipe(P);
    float *red = reinterpret_cast<float *>(const_cast<uint8_t *>(reinterpret_cast<const uint8_t *>(&P)) + P.off_red);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int wt = KS2 ? warp >> 1 : warp, nwt = KS2 ? 4 : 8;
    const bool fin = !KS2 || (warp & 1) == 0;  // this warp finishes its tiles
    float sc[TPW][2], bs[TPW][2], iv[TPW][2];
    if (fin) {  // fetched while the products run
        const float *ps = L.s, *pb = L.b, *pi = L.inv;
        const float sx = L.sx;
#pragma unroll
        for (int i = 0; i < TPW; i++)
#pragma unroll
            for (int hr = 0; hr < 2; hr++) {
                const int nl = (wt + nwt * i) * 16 + g + 8 * hr, n = base + nl + nl / HC * seg;
                sc[i][hr] = __fmul_rn(sx, __ldg(ps + n));
                bs[i][hr] = __ldg(pb + n);
                iv[i][hr] = Q8 ? __ldg(pi + n) : 0.0f;
            }
    }
    const int8_t *ap = act + g * stride + 16 * t;
    int nkb = (KS2 ? K >> 1 : K) >> 6;
    if (KS2) ap += (warp & 1) * nkb * 64;
    float acc[TPW][NB][4];
    if (KS2) {
        dr_gemm<NB, TPW>(ap, stride, nkb, pp.ring, pp.full, pp.empty, pp.slots, it, pp.wait, acc);
        float4 *rp = reinterpret_cast<float4 *>(red) + (size_t)wt * TPW * NB * 32 + lane;
        if (!fin) {
#pragma unroll
            for (int i = 0; i < TPW; i++)
#pragma unroll
                for (int nt = 0; nt < NB; nt++)
                    rp[(i * NB + nt) * 32] = make_float4(acc[i][nt][0], acc[i][nt][1], acc[i][nt][2], acc[i][nt][3]);
        }
        dr_sync();
        if (!fin) return;
#pragma unroll
        for (int i = 0; i < TPW; i++)
#pragma unroll
            for (int nt = 0; nt < NB; nt++) {
                const float4 v = rp[(i * NB + nt) * 32];  // both halves exact: the sum is fl(acc)
                acc[i][nt][0] = __fadd_rn(acc[i][nt][0], v.x);
                acc[i][nt][1] = __fadd_rn(acc[i][nt][1], v.y);
                acc[i][nt][2] = __fadd_rn(acc[i][nt][2], v.z);
                acc[i][nt][3] = __fadd_rn(acc[i][nt][3], v.w);
            }
    } else if (TPW > 1) {
        dr_gemm<NB, TPW>(ap, stride, nkb, pp.ring, pp.full, pp.empty, pp.slots, it, pp.wait, acc);  // K <= 512
    } else {
        // 1024 products at a time stay exact; the sum of two is fl(acc)
        float hi[TPW][NB][4];
#pragma unroll
        for (int nt = 0; nt < NB; nt++)
#pragma unroll
            for (int q = 0; q < 4; q++) acc[0][nt][q] = 0.0f;
#pragma unroll 1
        for (; nkb > 0; nkb -= 16, ap += 1024) {
            dr_gemm<NB, TPW>(ap, stride, min(nkb, 16), pp.ring, pp.full, pp.empty, pp.slots, it, pp.wait, hi);
#pragma unroll
            for (int nt = 0; nt < NB; nt++)
#pragma unroll
                for (int q = 0; q < 4; q++) acc[0][nt][q] = __fadd_rn(acc[0][nt][q], hi[0][nt][q]);
        }
    }
#pragma unroll
    for (int i = 0; i < TPW; i++)
#pragma unroll
        for (int nt = 0; nt < NB; nt++)
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int hr = q >> 1, n = (wt + nwt * i) * 16 + g + 8 * hr, row = nt * 8 + 2 * t + (q & 1);
                const float y = __fadd_rn(__fmul_rn(acc[i][nt][q], sc[i][hr]), bs[i][hr]);
                if (!Q8) reinterpret_cast<float *>(dst)[row * ldo + n] = y;
                else dst[row * ldo + n] = (uint8_t)q8_bits(relu && !(y > 0.0f) ? 0.0f : y, iv[i][hr]);
            }
}

// nearest float to S 2^e / d, the common case (d a power of two, a normal
// result) inline
__device__ __noinline__ float dr_rn32_general(long long S, int e, int kd, unsigned z, unsigned long long zm) {
    return rn32_scaled_mul(S, e, kd, z, zm);
}
MNMT_DEV float dr_rn32(long long S, int e, const DrParams &P) {
    if (P.ln_dodd == 1 && S != 0) {
        const uint32_t b = __float_as_uint(ll2float(S));
        const int fe = (int)((b >> 23) & 0xFFu) + e - P.ln_kd;
        if (fe >= 1 && fe <= 254) return __uint_as_float(b + ((uint32_t)(e - P.ln_kd) << 23));
    }
    return dr_rn32_general(S, e, P.ln_kd, (unsigned)P.ln_dodd, P.ln_zm);
}
__device__ __noinline__ long long dr_fx_scale(float v, int shift) { return fx_scale(v, shift); }

// Attention of AR rows of one head by a warp: attn_core's arithmetic in compact
// loops over (32 keys, set of rows that reads them).  A row's position j lives at
// kc / vc + (base[b] + prow[b][j]) rs + 64 j; `same` has a bit per 16 keys at
// which the rows read the same keys and values.  Z comes out of the products
// too, as one more column tile of ones.  The codes go to the first nc CTAs.
// Bound by the latency of each step's loads and chains (two warps a scheduler):
// with a lane per key and a row after the other, 102 to 124 keys of 4 rows took
// 8.5 thousand cycles of scores, 4 to 6.5 of softmax and 11 to 14 of values, in
// steps of 32 keys and all rows 6.2, 2.1 and 8.2 (512 rows, d = 512: 601 us a
// step -> 569; 256 rows 542 -> 509; greedy, 128 rows, 495 -> 445).
template <int AR>
__device__ __noinline__ void dr_attention(const DrParams &P, const int8_t *q, int q_ld, int nb, int n, float sigma, float rho,
                                          int *sc, const int8_t *kc, const int8_t *vc, size_t rs, const int *base,
                                          const uint8_t *prow, uint32_t same, uint32_t out, int out_ld, uint32_t xbar, int nc) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, cap = P.cap;
    auto at = [&](int j, int b) {
        return (size_t)((base ? base[b] : 0) + (prow ? (int)prow[b * cap + j] : 0)) * rs + (size_t)j * 64;
    };
    float mine = -INFINITY;  // lane b: row b's maximum
    {
        // Four lanes read a key (whole lines per load), 8 keys a load; the sum
        // scattered over the four leaves lane (g, t) with key 8 t + g of 32.
        // Every step scores the keys against all rows, in one straight run of
        // independent sums, and keeps those of the rows that read these keys.
        float mx[AR];
        int4 qr[AR], nx[4];
#pragma unroll
        for (int b = 0; b < AR; b++) {
            mx[b] = -INFINITY;
            qr[b] = *reinterpret_cast<const int4 *>(q + (b < nb ? b : 0) * q_ld + 16 * t);
        }
        auto kload = [&](int j0, int b) {
#pragma unroll
            for (int i = 0; i < 4; i++) nx[i] = *reinterpret_cast<const int4 *>(kc + at(min(j0 + 8 * i + g, n - 1), b) + 16 * t);
        };
        kload(0, 0);
        int j0 = 0, b = 0;
#pragma unroll 1
        while (j0 < n) {
            int4 kr[4];
#pragma unroll
            for (int i = 0; i < 4; i++) kr[i] = nx[i];
            const bool one = AR == 1 || ((same >> (j0 >> 4)) & 3u) == 3u, next = one || b + 1 == nb;
            const int j1 = next ? j0 + 32 : j0, b1 = next ? 0 : b + 1, j = j0 + 8 * t + g;
            if (j1 < n) kload(j1, b1);  // the next keys are on their way during this step
#pragma unroll
            for (int r = 0; r < AR; r++) {
                int acc[4];
#pragma unroll
                for (int i = 0; i < 4; i++) acc[i] = dot16(qr[r], kr[i], 0);
                gemv_reduce<4, 4>(acc, t);
                const float s = __fmul_rn(__int2float_rn(acc[0]), sigma);
                if (j < n && (one || r == b)) {
                    sc[r * cap + j] = __float_as_int(s);
                    mx[r] = fmaxf(mx[r], s);
                }
            }
            j0 = j1;
            b = b1;
        }
#pragma unroll
        for (int r = 0; r < AR; r++) {
            const float m = warp_max_f(mx[r]);
            if (lane == r) mine = m;
        }
    }
    __syncwarp();
    const int n16 = (n + 15) & ~15;
    {
        float m[AR];
#pragma unroll
        for (int r = 0; r < AR; r++) m[r] = __shfl_sync(0xFFFFFFFFu, mine, r);
#pragma unroll 1
        for (int j = lane; j < n16; j += 32) {  // the rows' chains of one key run side by side
            float v[AR];
#pragma unroll
            for (int r = 0; r < AR; r++) v[r] = __int_as_float(sc[r * cap + j]);
#pragma unroll
            for (int r = 0; r < AR; r++) {
                const int w = softmax_weight(__fsub_rn(v[r], m[r]));
                sc[r * cap + j] = j < n ? w : 0;
            }
        }
    }
    __syncwarp();
    float acc[9][4];
#pragma unroll
    for (int j = 0; j < 9; j++)
#pragma unroll
        for (int i = 0; i < 4; i++) acc[j][i] = 0.0f;
    const int qb = g & 3, sh = g >= 4 ? 8 : 0;
    const int *er = sc + (qb < nb ? qb : 0) * cap + 4 * t;
    uint2 nx[8];
    auto vload = [&](int j0, int b) {
#pragma unroll
        for (int i = 0; i < 8; i++)  // past the end: weight 0
            nx[i] = *reinterpret_cast<const uint2 *>(vc + at(min(j0 + 16 * (i >> 2) + 4 * t + (i & 3), n - 1), b) + 8 * g);
    };
    vload(0, 0);
    int j0 = 0, b = 0;
#pragma unroll 1
    while (j0 < n) {
        uint2 raw[8];
#pragma unroll
        for (int i = 0; i < 8; i++) raw[i] = nx[i];
        const bool one = AR == 1 || ((same >> (j0 >> 4)) & 3u) == 3u, next = one || b + 1 == nb;
        const int j1 = next ? j0 + 32 : j0, b1 = next ? 0 : b + 1;
        if (j1 < n) vload(j1, b1);  // the next values are on their way during this step
        const bool in = qb < nb && (one || qb == b);
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const bool inh = in && j0 + 16 * h < n16;
            const uint32_t k01 = inh ? 0x00FF00FFu : 0u, k2 = inh && g < 4 ? 0x01FF01FFu : 0u;
            const int4 e = *reinterpret_cast<const int4 *>(er + min(j0 + 16 * h, n16 - 16));
            uint32_t a[4];
            a[0] = half2_sub_1024((__byte_perm((uint32_t)e.x >> sh, (uint32_t)e.y >> sh, 0x5410) & k01) | 0x64006400u);
            a[2] = half2_sub_1024((__byte_perm((uint32_t)e.z >> sh, (uint32_t)e.w >> sh, 0x5410) & k01) | 0x64006400u);
            a[1] = half2_sub_1024((__byte_perm((uint32_t)e.x, (uint32_t)e.y, 0x7632) & k2) | 0x64006400u);
            a[3] = half2_sub_1024((__byte_perm((uint32_t)e.z, (uint32_t)e.w, 0x7632) & k2) | 0x64006400u);
            mma_f16_16816(acc[8], a, 0x3C003C00u, 0x3C003C00u);
#pragma unroll
            for (int w = 0; w < 2; w++) {
                uint32_t u[4], bq[4][2];
#pragma unroll
                for (int i = 0; i < 4; i++) u[i] = (w ? raw[4 * h + i].y : raw[4 * h + i].x) ^ 0x80808080u;
#pragma unroll
                for (int p = 0; p < 2; p++) {
                    const uint32_t lo = __byte_perm(u[2 * p], u[2 * p + 1], 0x5140), hi = __byte_perm(u[2 * p], u[2 * p + 1], 0x7362);
                    bq[0][p] = h2_sub(__byte_perm(lo, 0x64646464u, 0x4140), 0x64806480u);
                    bq[1][p] = h2_sub(__byte_perm(lo, 0x64646464u, 0x4342), 0x64806480u);
                    bq[2][p] = h2_sub(__byte_perm(hi, 0x64646464u, 0x4140), 0x64806480u);
                    bq[3][p] = h2_sub(__byte_perm(hi, 0x64646464u, 0x4342), 0x64806480u);
                }
#pragma unroll
                for (int x = 0; x < 4; x++) mma_f16_16816(acc[4 * w + x], a, bq[x][0], bq[x][1]);
            }
        }
        j0 = j1;
        b = b1;
    }
    // as in attn_rows: lanes g < 4 finish the elements 16 t + j of row g, lanes
    // g >= 4 those from 16 t + 8 of row g - 4; column tile 8 holds Z
    auto pieces = [&](const float (&x)[4], float &a0, float &a1, float &a2) {
        const float v1 = __shfl_xor_sync(0xFFFFFFFFu, g < 4 ? x[1] : x[0], 16), v2 = __shfl_xor_sync(0xFFFFFFFFu, x[3], 16);
        a0 = g < 4 ? x[0] : v1;
        a1 = g < 4 ? v1 : x[1];
        a2 = g < 4 ? x[2] : v2;
    };
    auto whole = [](float a0, float a1, float a2) {
        return (long long)__float2int_rn(a0) + (long long)__float2int_rn(a1) * 256 + (long long)__float2int_rn(a2) * 65536;
    };
    float z0, z1, z2;
    pieces(acc[8], z0, z1, z2);
    const float iz = softmax_inv(__fmaf_rn(z2, 65536.0f, __fmaf_rn(z1, 256.0f, z0)));  // two roundings, Z >= 2^24
    const float slack = __fmul_rn(fabsf(rho), 0x1p-15f);
    uint32_t words[2] = {0u, 0u};
#pragma unroll
    for (int j = 0; j < 8; j++) {
        float a0, a1, a2;
        pieces(acc[j], a0, a1, a2);
        const float fn = __fmaf_rn(a2, 65536.0f, __fmaf_rn(a1, 256.0f, a0));
        float c = 0.0f;
        if (qb < nb)
            c = q8_context(fn, iz, rho, slack, [&]() { return att_ctx_exact(whole(a0, a1, a2), whole(z0, z1, z2), rho); });
        words[j >> 2] |= (__float_as_uint(__fadd_rn(c, 12582912.0f)) & 0xFFu) << (8 * (j & 3));
    }
    if (qb < nb) {
        const uint32_t local = out + (uint32_t)(qb * out_ld + 16 * t + (g >= 4 ? 8 : 0));
        for (int k = 0; k < nc; k++) dr_send2(dr_mapa(local, k), words[0], words[1], dr_mapa(xbar, k));
    }
    __syncwarp();
}

// LayerNorm of one owned row by wpr warps (part 0 .. wpr - 1, EPL elements per
// lane: element part d / wpr + 32 i + lane), the arithmetic of warp_layernorm.
// With y, the residual first takes the linear's output, r = fl(fl(gamma r) + y),
// once that has arrived (bar, par; then re-armed for `arm` bytes).  Partial
// extremes and sums meet in `part_s` behind the row's named barrier; the centred
// row's largest magnitude follows from the extremes (subtraction is monotone).
// Leaves the codes of the row in `codes`, behind a last barrier.  False if the
// wait has given up.
struct DrLnRow {
    float *r;
    const float *y;
    uint32_t *part_s;  // [8] amax, [8] max, [8] min, then [2][8] int64 sums
    int8_t *codes;
    int part, wpr, slot;
    bool live;
};
template <int EPL>
__device__ __noinline__ bool dr_layernorm(const DrParams &P, const DrLnRow w, const float *gp, const float *bp, float inv,
                                          float gamma, const DrWait wait, uint32_t bar, uint32_t par, uint32_t arm) {
    const int lane = threadIdx.x & 31, e0 = w.part * (P.d / w.wpr) + lane;
    auto sync = [&]() {
        if (w.wpr == 1) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(2 + w.slot), "r"(w.wpr * 32) : "memory");
    };
    float gv[EPL], bv[EPL], v[EPL];
#pragma unroll
    for (int i = 0; i < EPL; i++) {
        gv[i] = __ldg(gp + e0 + 32 * i);
        bv[i] = __ldg(bp + e0 + 32 * i);
        v[i] = w.live ? w.r[e0 + 32 * i] : 0.0f;
    }
    bool ok = true;
    if (bar) {
        ok = wait(bar, par);
        if (threadIdx.x == 0 && arm && ok) mbar_expect_tx(bar, arm);
    }
    if (!w.live) return ok;
    unsigned am = 0, hi = 0, lo = 0xFFFFFFFFu;
#pragma unroll
    for (int i = 0; i < EPL; i++) {
        if (w.y) {
            v[i] = __fadd_rn(__fmul_rn(gamma, v[i]), w.y[e0 + 32 * i]);
            w.r[e0 + 32 * i] = v[i];
        }
        const unsigned o = ordered_bits(v[i]);
        am = max(am, __float_as_uint(v[i]) & 0x7FFFFFFFu);
        hi = max(hi, o);
        lo = min(lo, o);
    }
    am = __reduce_max_sync(0xFFFFFFFFu, am);
    hi = __reduce_max_sync(0xFFFFFFFFu, hi);
    lo = __reduce_min_sync(0xFFFFFFFFu, lo);
    long long *sum_s = reinterpret_cast<long long *>(w.part_s + 24);
    if (w.wpr > 1) {
        if (lane == 0) {
            w.part_s[w.part] = am;
            w.part_s[8 + w.part] = hi;
            w.part_s[16 + w.part] = lo;
        }
        sync();
        for (int k = 0; k < w.wpr; k++) {
            am = max(am, w.part_s[k]);
            hi = max(hi, w.part_s[8 + k]);
            lo = min(lo, w.part_s[16 + k]);
        }
    }
    const float amax = __uint_as_float(am);
    if (!(amax < 0x1p32f) && lane == 0) set_status(P.status, MNMT_EOVERFLOW);
    const int ea = exp_bound(amax);
    auto total = [&](long long x, int which) {
        x = warp_sum_exact(x);
        if (w.wpr == 1) return x;
        if (lane == 0) sum_s[8 * which + w.part] = x;
        sync();
        x = 0;
        for (int k = 0; k < w.wpr; k++) x += sum_s[8 * which + k];
        return x;
    };
    long long s1 = 0;
    if (ea >= -70 && ea <= 33) {
        s1 = fx_sum<EPL>(v, ea);
    } else {
#pragma unroll 1
        for (int i = 0; i < EPL; i++) s1 += dr_fx_scale(w.r[e0 + 32 * i], 52 - ea);
    }
    const float mu = dr_rn32(total(s1, 0), ea - 52, P);
    const int eb = exp_bound(fmaxf(fabsf(__fsub_rn(from_ordered_bits(hi), mu)), fabsf(__fsub_rn(from_ordered_bits(lo), mu))));
#pragma unroll
    for (int i = 0; i < EPL; i++) v[i] = __fsub_rn(v[i], mu);
    long long s2 = 0;
    if (eb >= -36 && eb <= 34) {
        float c2[EPL];
        const float su = __uint_as_float((uint32_t)(127 - eb) << 23);
#pragma unroll
        for (int i = 0; i < EPL; i++) {
            const float cc = __fmul_rn(v[i], su);
            c2[i] = __fmul_rn(cc, cc);
        }
        s2 = fx_sum<EPL>(c2, 0);
    } else {
#pragma unroll 1
        for (int i = 0; i < EPL; i++) {
            const float cc = __fsub_rn(w.r[e0 + 32 * i], mu);
            s2 += dr_fx_scale(__fmul_rn(cc, cc), 52 - 2 * eb);
        }
    }
    const float var = dr_rn32(total(s2, 1), 2 * eb - 52, P);
    const float rstd = __fdiv_rn(1.0f, __fsqrt_rn(__fadd_rn(var, 1e-5f)));
#pragma unroll
    for (int i = 0; i < EPL; i++)
        w.codes[e0 + 32 * i] = (int8_t)q8_bits(__fadd_rn(__fmul_rn(__fmul_rn(v[i], rstd), gv[i]), bv[i]), inv);
    sync();
    return ok;
}

// One warp: the caches that layer l's attention of these rows and heads reads,
// to L2.  Caches larger than L2 do not stay there from step to step, and the
// attention waits for every step of its loads (512 rows 568 -> 555 us a step, 256
// rows 509 -> 495, greedy 128 rows 444 -> 411; where they stay, 1 % slower).  Not
// a beam's own keys and values: their rows scatter (559).
__device__ __noinline__ void dr_prefetch_layer(const DrParams &P, int l, int r0, int rows, int head0, int heads) {
    const DrLayer &Y = P.layer[l];
    const int lane = threadIdx.x & 31, s0 = r0 / P.beam, ns = (r0 + rows - 1) / P.beam - s0 + 1, t = *P.t_ptr, per = 2 * heads;
    for (int k = lane; k < ns * per; k += 32) {
        const int sent = s0 + k / per, head = head0 + (k % per >> 1), len = P.src_len[sent];
        dr_prefetch((k & 1 ? Y.cross_v : Y.cross_k) + ((size_t)sent * P.H + head) * P.S * 64,
                    64 * (len < 1 ? 1 : (len > P.S ? P.S : len)));
    }
    for (int k = lane; P.beam == 1 && t > 0 && k < rows * per; k += 32) {
        const int row = r0 + k / per, head = head0 + (k % per >> 1);
        dr_prefetch((k & 1 ? Y.self_v : Y.self_k) + ((size_t)row * P.H + head) * P.T * 64, t * 64);
    }
}

// NB: the cluster takes 8 NB rows; HPC: heads per CTA (the cluster has H / HPC)
template <int NB, int HPC>
__global__ void __launch_bounds__(DR_THREADS, 1) decode_rows_kernel(const DrParams *__restrict__ Pp) {
    pdl_grid_wait();
    if (*Pp->done) return;  // uniform over the grid
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr int RB = 8 * NB, HC = 64 * HPC;
    constexpr int AR = NB * HPC < 4 ? NB * HPC : 4;  // rows of a head that a warp attends for at a time
    {
        const int n16 = Pp->param_bytes / 16;
        for (int i = threadIdx.x; i < n16; i += DR_THREADS)
            reinterpret_cast<int4 *>(smem)[i] = reinterpret_cast<const int4 *>(Pp)[i];
    }
    __syncthreads();
    const DrParams &P = *reinterpret_cast<const DrParams *>(smem);
    const int d = P.d, H = P.H, F = P.F, T = P.T, nc = P.nc, c = (int)(blockIdx.x % (unsigned)nc);
    const int r0 = (int)(blockIdx.x / (unsigned)nc) * RB;  // the cluster's first row
    const int rows = min(RB, P.R - r0);                    // its valid rows
    const int own0 = c * RB / nc, own1 = (c + 1) * RB / nc;  // the rows this CTA owns
    const int slots = P.slots;
    const uint32_t bars = dr_smem(smem + P.off_bar), full = bars, empty = bars + 8u * DR_MAX_SLOTS,
                   xbars = empty + 8u * DR_MAX_SLOTS;
    volatile uint32_t *abort_flag = dr_abort(P);
    const int nx = 9 * P.n_dec;
    auto xbytes = [&](int x) -> uint32_t {
        const int k = dr_exchange_kind(x);
        return (uint32_t)(k == DX_Y ? (own1 - own0) * d * 4 : (k == DX_H ? RB * F : RB * d));
    };
    if (threadIdx.x == 0) {
        for (int i = 0; i < slots; i++) {
            mbar_init(full + 8u * i, 1);
            mbar_init(empty + 8u * i, DR_WARPS);
        }
        mbar_init(xbars, 1);
        mbar_init(xbars + 8u, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int i = 0; i < 2; i++) mbar_expect_tx(xbars + 8u * i, xbytes(i));
    }
    __syncthreads();
    // every CTA's barriers are set before any remote store (waited for below)
    asm volatile("barrier.cluster.arrive.release;\n" ::: "memory");
    const DrWait wait{P.status, abort_flag};
    uint8_t *ring = smem + P.off_ring;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (warp == DR_WARPS) {
        // ---- producer: the CTA's weight stream through the ring ----
        const uint8_t *src = P.stream + (size_t)c * P.stream_cta;
        const uint32_t n = (uint32_t)(P.stream_cta / DR_SLOT);
        uint32_t s = 0, par = 1, i = 0;
        auto feed = [&](uint32_t end) {  // one thread: slots up to `end`; false after a timed-out wait
            for (; i < end; i++) {
                // (the flag after the wait: warps that have given up pass slots unread)
                if (i >= (uint32_t)slots && (!wait(empty + 8u * s, par) || *abort_flag)) return false;
                mbar_expect_tx(full + 8u * s, DR_SLOT);
                bulk_load(dr_smem(ring + s * DR_SLOT), src + (size_t)i * DR_SLOT, DR_SLOT, full + 8u * s);
                if (++s == (uint32_t)slots) {
                    s = 0;
                    par ^= 1;
                }
            }
            return true;
        };
        if (!P.far_caches) {
            if (lane == 0) feed(n);
        } else {
            bool ok = true;
            for (int l = 0; l < P.n_dec && ok; l++) {
                dr_prefetch_layer(P, l, r0, rows, c * HPC, HPC);
                if (lane == 0) ok = feed(n / (uint32_t)P.n_dec * (uint32_t)(l + 1));
                ok = __shfl_sync(0xFFFFFFFFu, ok, 0);
            }
        }
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory");
        dr_sync_all();  // the compute warps are through
        if (*abort_flag) {
            // the copies in flight land (bounded) before the CTA ends
            if (lane == 0)
                for (uint32_t k = i > (uint32_t)slots ? i - slots : 0; k < i; k++) mbar_wait(full + 8u * (k % slots), (k / slots) & 1);
            __syncwarp();
            dr_leave();
        }
        return;
    }

    // ---- compute warps ----
    int8_t *actA = reinterpret_cast<int8_t *>(smem + P.off_a);   // [RB][d + pad] LayerNorm codes
    int8_t *actC = reinterpret_cast<int8_t *>(smem + P.off_h);   // [RB][d + pad] context, or
    int8_t *actH = actC;                                         // [RB][F + pad] FFN hidden (never live together)
    float *ybuf = reinterpret_cast<float *>(smem + P.off_y);     // [own rows][d] linear outputs of the owned rows
    float *rbuf = reinterpret_cast<float *>(smem + P.off_r);     // [own rows][d] residual
    int8_t *qbuf = reinterpret_cast<int8_t *>(smem + P.off_q);   // [RB][HC] queries of the CTA's heads
    float *red = reinterpret_cast<float *>(smem + P.off_red);    // K-half partials; attention weights
    uint8_t *stage = smem + P.off_stage;                         // [RB][.] outputs on their way out
    uint8_t *prow = smem + P.off_prow;                           // [RB][cap]
    int *meta = reinterpret_cast<int *>(smem + P.off_meta);      // [RB] token, [RB] sentence's first row, [RB] owner, [8] same-row masks
    uint8_t *lns = smem + P.off_ln;                              // [8] row slots: 256 bytes of partials, d codes
    const int sa = P.stride_a, sh = P.stride_h;
    const int t = *P.t_ptr, cap = P.cap;
    for (int r = threadIdx.x; r < RB; r += DR_WARPS * 32) {
        const int rg = r0 + r;
        int id = r < rows ? P.tok[rg] : 0;
        if (id < 0 || id >= P.V) {
            set_status(P.status, MNMT_EINVAL);
            id = 0;
        }
        meta[r] = id;
        meta[RB + r] = rg / P.beam * P.beam;
        int o = 0;
        while ((o + 1) * RB / nc <= r) o++;
        meta[2 * RB + r] = o;
    }
    // physical rows of every position, as offsets in the sentence
    if (P.beam > 1) {
        for (int j = lane; j <= t; j += 32) {
#pragma unroll
            for (int k = 0; k < NB; k++) {
                const int r = warp + 8 * k, rg = r0 + r, base = rg / P.beam * P.beam;
                if (r < rows) prow[r * cap + j] = (uint8_t)(j < t ? P.anc[(size_t)rg * T + j] - base : rg - base);
            }
        }
    }
    dr_sync();
    // positions at which a chunk of AR rows reads one physical row: a bit per 16 keys
    if (P.beam > 1 && warp < RB / AR) {
        const int c0 = warp * AR, nb = min(AR, max(0, rows - c0)), nk = t + 1;
        uint32_t same = nb > 1 ? 0u : 0xFFFFFFFFu;
        if (nb > 1)
            for (int kb = 0; kb * 16 < nk; kb++) {
                const int j = min(kb * 16 + (lane & 15), nk - 1);
                bool eq = true;
                for (int b = 1; b < nb; b++)
                    eq = eq && meta[RB + c0] + prow[c0 * cap + j] == meta[RB + c0 + b] + prow[(c0 + b) * cap + j];
                if (__all_sync(0xFFFFFFFFu, eq)) same |= 1u << kb;
            }
        if (nb > 1 && nk <= 16 * 31) same |= 0xFFFFFFFFu << ((nk + 15) >> 4);  // no keys there
        if (lane == 0) meta[3 * RB + warp] = (int)same;
    }

    // ---- embedding of the owned rows ----
    const int nown = own1 - own0;
    if (P.proj_w) {
        const int ec = P.E / 16;
        for (int i = threadIdx.x; i < nown * d; i += DR_WARPS * 32) {
            const int rr = i / d, n = i - rr * d, id = meta[own0 + rr];
            const int4 *q = reinterpret_cast<const int4 *>(P.emb_q + (size_t)id * P.E);
            const int4 *w = reinterpret_cast<const int4 *>(P.proj_w + (size_t)n * P.E);
            const float es = P.emb_s[id], ps = P.proj_s[n], pb = P.proj_b[n], pe = P.pe[(size_t)t * d + n];
            int a = 0;
#pragma unroll 8
            for (int k = 0; k < ec; k++) a = dot16(__ldg(q + k), __ldg(w + k), a);
            rbuf[i] = __fadd_rn(__fmul_rn(dequant_bias(a, es, ps, pb), P.emb_scale), pe);
        }
    } else {
#pragma unroll 2
        for (int i = threadIdx.x; i < nown * d / 4; i += DR_WARPS * 32) {
            const int rr = i / (d / 4), n = 4 * (i - rr * (d / 4)), id = meta[own0 + rr];
            const char4 q = *reinterpret_cast<const char4 *>(P.emb_q + (size_t)id * P.E + n);
            const float4 pe = *reinterpret_cast<const float4 *>(P.pe + (size_t)t * d + n);
            const float es = P.emb_s[id], sc = P.emb_scale;
            *reinterpret_cast<float4 *>(rbuf + 4 * i) = make_float4(
                __fadd_rn(__fmul_rn(__fmul_rn((float)q.x, es), sc), pe.x), __fadd_rn(__fmul_rn(__fmul_rn((float)q.y, es), sc), pe.y),
                __fadd_rn(__fmul_rn(__fmul_rn((float)q.z, es), sc), pe.z), __fadd_rn(__fmul_rn(__fmul_rn((float)q.w, es), sc), pe.w));
        }
    }
    dr_sync();
    asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory");

    int x = 0;        // exchanges so far
    int live = nc;    // CTAs that this thread sends to: all, or none after a timed-out wait
    uint32_t it = 0;  // ring slots so far
    // wait for exchange x's bytes; arm its barrier for exchange x + 2
    auto receive = [&]() {
        const uint32_t bar = xbars + 8u * (uint32_t)(x & 1);
        const bool ok = live && wait(bar, (uint32_t)(x >> 1) & 1u);
        if (!ok) live = 0;
        if (threadIdx.x == 0 && x + 2 < nx && ok) mbar_expect_tx(bar, xbytes(x + 2));
        x++;
    };
    // LayerNorm of the owned rows, 2^ln_w warps per row; add: after the linear
    // whose outputs exchange x brings.  The codes go to every CTA (last: to
    // memory, with the residual).
    auto ln_rows = [&](const float *gp, const float *bp, float inv, bool add, float gamma, bool last) {
        const int lw = P.ln_w, wpr = 1 << lw, slot = warp >> lw, part = warp & (wpr - 1), gt = threadIdx.x & (wpr * 32 - 1);
        uint32_t bar = 0, par = 0, arm = 0;
        if (add) {
            bar = live ? xbars + 8u * (uint32_t)(x & 1) : 0u;
            par = (uint32_t)(x >> 1) & 1u;
            arm = x + 2 < nx ? xbytes(x + 2) : 0u;
            x++;
        }
        const uint32_t xbar = xbars + 8u * (uint32_t)(x & 1);
        for (int rr = slot; rr < nown || (rr == slot && bar); rr += DR_WARPS >> lw) {
            uint8_t *ls = lns + slot * (256 + d);
            const DrLnRow w{rbuf + (size_t)rr * d, add ? ybuf + (size_t)rr * d : nullptr, reinterpret_cast<uint32_t *>(ls),
                            reinterpret_cast<int8_t *>(ls + 256), part, wpr, slot, rr < nown};
            bool ok;
            switch (P.ln_epl) {
                case 2: ok = dr_layernorm<2>(P, w, gp, bp, inv, gamma, wait, bar, par, arm); break;
                case 3: ok = dr_layernorm<3>(P, w, gp, bp, inv, gamma, wait, bar, par, arm); break;
                case 4: ok = dr_layernorm<4>(P, w, gp, bp, inv, gamma, wait, bar, par, arm); break;
                case 6: ok = dr_layernorm<6>(P, w, gp, bp, inv, gamma, wait, bar, par, arm); break;
                case 8: ok = dr_layernorm<8>(P, w, gp, bp, inv, gamma, wait, bar, par, arm); break;
                case 12: ok = dr_layernorm<12>(P, w, gp, bp, inv, gamma, wait, bar, par, arm); break;
                default: ok = dr_layernorm<16>(P, w, gp, bp, inv, gamma, wait, bar, par, arm); break;
            }
            if (!ok) live = 0;
            bar = 0;
            if (rr >= nown) break;
            const int row = own0 + rr, rg = r0 + row, chunks = d >> 4;
            if (last) {
                if (row < rows) {
                    for (int k = gt; k < chunks; k += wpr * 32) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(ls + 256 + 16 * k);
                        const size_t o = (size_t)rg * d + 16 * k;
                        *reinterpret_cast<uint4 *>(P.act_out + o) = v;
                        if (P.act16_out) {
                            uint32_t h[8];
                            codes_to_half2((int)v.x, h[0], h[1]);
                            codes_to_half2((int)v.y, h[2], h[3]);
                            codes_to_half2((int)v.z, h[4], h[5]);
                            codes_to_half2((int)v.w, h[6], h[7]);
                            reinterpret_cast<uint4 *>(P.act16_out + o)[0] = make_uint4(h[0], h[1], h[2], h[3]);
                            reinterpret_cast<uint4 *>(P.act16_out + o)[1] = make_uint4(h[4], h[5], h[6], h[7]);
                        }
                    }
                    for (int k = gt; k < d / 4; k += wpr * 32)
                        reinterpret_cast<float4 *>(P.resid_out + (size_t)rg * d)[k] =
                            reinterpret_cast<const float4 *>(rbuf + (size_t)rr * d)[k];
                }
            } else {
                const int per = wpr * 32 / chunks, q0 = gt / chunks, ch = gt - q0 * chunks;  // CTAs served at a time
                if (q0 < per) {
                    const uint4 v = *reinterpret_cast<const uint4 *>(ls + 256 + 16 * ch);
                    const uint32_t local = dr_smem(actA + (size_t)row * sa + 16 * ch);
                    for (int q = q0; q < live; q += per) dr_send4(dr_mapa(local, q), v, dr_mapa(xbar, q));
                }
            }
            if (rr + (DR_WARPS >> lw) < nown) {  // the slot's partials and codes are free again
                if (wpr == 1) __syncwarp();
                else asm volatile("bar.sync %0, %1;" ::"r"(2 + slot), "r"(wpr * 32) : "memory");
            }
        }
    };
    // the CTA's HC columns of a residual linear: to the owners of the rows
    auto send_y = [&]() {
        dr_sync();
        const uint32_t xbar = xbars + 8u * (uint32_t)(x & 1);
        const float *sy = reinterpret_cast<const float *>(stage);
        for (int i = threadIdx.x; i < RB * HC / 4 && live; i += DR_WARPS * 32) {
            const int row = i / (HC / 4), ch = i % (HC / 4), o = meta[2 * RB + row];
            const uint4 v = *reinterpret_cast<const uint4 *>(sy + row * (HC + 4) + 4 * ch);
            const uint32_t local = dr_smem(ybuf + (size_t)(row - o * RB / nc) * d + HC * c + 4 * ch);
            dr_send4(dr_mapa(local, o), v, dr_mapa(xbar, o));
        }
    };
    // attention of the CTA's heads; the codes go to every CTA's context buffer
    auto attend = [&](const DrLayer &Y, bool cross) {
        int *scw = reinterpret_cast<int *>(red) + (size_t)warp * AR * cap;
        const uint32_t xbar = xbars + 8u * (uint32_t)(x & 1);
        for (int item = warp; item < HPC * RB / AR; item += DR_WARPS) {
            const int hl = item / (RB / AR), head = c * HPC + hl, ck = item % (RB / AR), c0 = ck * AR;
            const int wnb = min(AR, max(0, rows - c0));  // the chunk's valid rows
            const uint32_t out = dr_smem(actC + (size_t)c0 * sa + 64 * head);
            // sets of rows that one call takes: beams of a sentence (or all
            // rows, through the ancestry table)
            for (int b0 = 0; b0 < wnb;) {
                const int rg = r0 + c0 + b0;
                int b1 = wnb, n = t + 1;
                const int8_t *kc = Y.self_k + (size_t)head * T * 64, *vc = Y.self_v + (size_t)head * T * 64;
                size_t rs = (size_t)H * T * 64;
                const int *base = meta + RB + c0;
                const uint8_t *pr = prow + c0 * cap;
                uint32_t same = (uint32_t)meta[3 * RB + ck];
                if (cross) {
                    const int sent = rg / P.beam;
                    b1 = min(wnb, b0 + (sent + 1) * P.beam - rg);
                    n = P.src_len[sent];
                    n = n < 1 ? 1 : (n > P.S ? P.S : n);
                    const size_t o = ((size_t)sent * H + head) * P.S * 64;
                    kc = Y.cross_k + o;
                    vc = Y.cross_v + o;
                } else if (P.beam == 1) {
                    b1 = b0 + 1;
                    kc += (size_t)rg * rs;
                    vc += (size_t)rg * rs;
                }
                if (cross || P.beam == 1) {
                    rs = 0;
                    base = nullptr;
                    pr = nullptr;
                    same = 0xFFFFFFFFu;
                }
                auto run = [&](auto rows_c) {
                    dr_attention<decltype(rows_c)::value>(P, qbuf + (c0 + b0) * HC + hl * 64, HC, b1 - b0, n,
                                                          cross ? Y.sigma2 : Y.sigma1, cross ? Y.rho2 : Y.rho1, scw, kc, vc, rs,
                                                          base, pr, same, out + (uint32_t)(b0 * sa), sa, xbar, live);
                };
                if (AR > 1 && b1 - b0 == 1) run(std::integral_constant<int, 1>{});
                else run(std::integral_constant<int, AR>{});
                b0 = b1;
            }
            // rows past the batch send zeros: every exchange has its full size
            for (int i = lane; i < (AR - wnb) * 8; i += 32) {
                const uint32_t local = out + (uint32_t)((wnb + (i >> 3)) * sa + 8 * (i & 7));
                for (int k = 0; k < live; k++) dr_send2(dr_mapa(local, k), 0u, 0u, dr_mapa(xbar, k));
            }
        }
    };
    constexpr int QT = 3, HT = 1;  // tiles per warp of QKV and of the 64 HPC wide linears
    constexpr bool K2 = HPC == 1;                 // ... on halves of K
    const int fc = F / nc, fst = fc + 16;
    // slots of a linear of `cols` columns and depth K
    auto used = [&](int cols, int K) { it += (uint32_t)(cols * K / DR_SLOT); };

    ln_rows(P.layer[0].ln1_g, P.layer[0].ln1_b, P.layer[0].inv_in1, false, 0.0f, false);
    receive();
    for (int i = 0; i < 3 * P.n_dec; i++) {
        const int l = i / 3, sub = i - 3 * l;  // self attention, cross attention, FFN
        const DrLayer &Y = P.layer[l];
        const DrLin &Lin = Y.lin[2 * sub], &Lout = Y.lin[2 * sub + 1];
        // ---- the sublayer's first linear ----
        if (sub == 0) {
            // queries stay, keys / values go into the cache
            constexpr int QS = 3 * HC + 16;
            dr_linear<NB, HC, QT, K2, true>(P, Lin, HC * c, d - HC, actA, sa, d, it, stage, QS, false);
            used(3 * HC, d);
            dr_sync();
            for (int k = threadIdx.x; k < RB * (3 * HC / 16); k += DR_WARPS * 32) {
                const int row = k / (3 * HC / 16), ch = k % (3 * HC / 16), seg = ch / (HC / 16), e = 16 * (ch % (HC / 16));
                const uint4 v = *reinterpret_cast<const uint4 *>(stage + row * QS + 16 * ch);
                if (seg == 0) {
                    *reinterpret_cast<uint4 *>(qbuf + row * HC + e) = v;
                } else if (row < rows) {
                    int8_t *dst = seg == 1 ? Y.self_k : Y.self_v;
                    *reinterpret_cast<uint4 *>(dst + (((size_t)(r0 + row) * H + c * HPC + e / 64) * T + t) * 64 + e % 64) = v;
                }
            }
        } else if (sub == 1) {
            dr_linear<NB, HC, HT, K2, true>(P, Lin, HC * c, 0, actA, sa, d, it, reinterpret_cast<uint8_t *>(qbuf), HC, false);
            used(HC, d);
        } else {
            if (HPC == 2 && fc == 512) dr_linear<NB, HC, 4, false, true>(P, Lin, fc * c, 0, actA, sa, d, it, stage, fst, true);
            else if (HPC == 2 && fc == 384) dr_linear<NB, HC, 3, false, true>(P, Lin, fc * c, 0, actA, sa, d, it, stage, fst, true);
            else if (fc == 256) dr_linear<NB, HC, 2, false, true>(P, Lin, fc * c, 0, actA, sa, d, it, stage, fst, true);
            else if (fc == 128) dr_linear<NB, HC, 1, false, true>(P, Lin, fc * c, 0, actA, sa, d, it, stage, fst, true);
            else if (HPC == 1 && fc == 192) dr_linear<NB, HC, 3, true, true>(P, Lin, fc * c, 0, actA, sa, d, it, stage, fst, true);
            else if (HPC == 1) dr_linear<NB, HC, 1, true, true>(P, Lin, fc * c, 0, actA, sa, d, it, stage, fst, true);
            used(fc, d);
        }
        dr_sync();
        if (sub < 2) {
            attend(Y, sub == 1);
        } else {
            const uint32_t xbar = xbars + 8u * (uint32_t)(x & 1);
            const int cpr = fc >> 4;  // 16-byte chunks per row
            for (int k = threadIdx.x; k < RB * cpr; k += DR_WARPS * 32) {
                const int row = k / cpr, ch = k - row * cpr;
                const uint4 v = *reinterpret_cast<const uint4 *>(stage + row * fst + 16 * ch);
                const uint32_t local = dr_smem(actH + (size_t)row * sh + c * fc + 16 * ch);
                for (int q = 0; q < live; q++) {
                    const int dst = c + q < nc ? c + q : c + q - nc;
                    dr_send4(dr_mapa(local, dst), v, dr_mapa(xbar, dst));
                }
            }
        }
        receive();
        // ---- its second linear, the residual and the next LayerNorm ----
        const int K2nd = sub < 2 ? d : F;
        dr_linear<NB, HC, HT, K2, false>(P, Lout, HC * c, 0, sub < 2 ? actC : actH, sub < 2 ? sa : sh, K2nd, it, stage, HC + 4, false);
        used(HC, K2nd);
        send_y();
        const bool last = i + 1 == 3 * P.n_dec;
        const DrLayer &Z = P.layer[last ? l : (sub == 2 ? l + 1 : l)];
        ln_rows(last ? P.fin_g : sub == 0 ? Z.ln2_g : sub == 1 ? Z.ln3_g : Z.ln1_g,
                last ? P.fin_b : sub == 0 ? Z.ln2_b : sub == 1 ? Z.ln3_b : Z.ln1_b,
                last ? P.inv_dout : sub == 0 ? Z.inv_in2 : sub == 1 ? Z.inv_in3 : Z.inv_in1, true, Lout.gam, last);
        if (!last) receive();
    }
    // unless a wait timed out: everything sent to this CTA has arrived (its last
    // exchange was received) and every weight copy was consumed; its own stores
    // carry their data
    dr_sync_all();
    if (*abort_flag) dr_leave();
}

const void *dr_kernel(int nb, int hpc) {
    if (hpc == 2) return (const void *)decode_rows_kernel<2, 2>;
    return nb == 1 ? (const void *)decode_rows_kernel<1, 1> : nb == 2 ? (const void *)decode_rows_kernel<2, 1>
                                                                      : (const void *)decode_rows_kernel<4, 1>;
}

cudaLaunchConfig_t dr_config(int nc, int clusters, size_t smem, cudaStream_t st, cudaLaunchAttribute *attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nc * clusters));
    cfg.blockDim = dim3(DR_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)nc;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

bool dr_shape_ok(int d, int H, int F, int E, int n_dec) {
    return H >= 2 && H <= 8 && H % 2 == 0 && d == 64 * H && F % (64 * H) == 0 && F / H <= 256 && F <= 2048 && E % 16 == 0 &&
           n_dec <= DR_LMAX;
}

size_t dr_bytes(int d, int F, int n_dec) { return (size_t)n_dec * ((size_t)6 * d * d + (size_t)2 * d * F); }

cudaError_t dr_pack(const DrPack &pk, int d, int H, int hpc, int F, uint8_t *out, cudaStream_t st) {
    const int nc = H / hpc;
    int most = 0;  // codes of a CTA's largest phase
    for (int p = 0; p < 6; p++) {
        const int n = dr_cols(p, hpc, F, nc) * (p == DR_W2 ? F : d);
        most = n > most ? n : most;
    }
    dr_pack_kernel<<<dim3((most / 16 * nc + 255) / 256, 6 * pk.n_dec), 256, 0, st>>>(pk, d, nc, hpc, F, out,
                                                                                 dr_bytes(d, F, pk.n_dec) / nc);
    return cudaGetLastError();
}

size_t dr_layout(DrParams &P, int nb, int hpc, size_t max_smem) {
    const int rb = 8 * nb, d = P.d, F = P.F, nc = P.H / hpc, fc = F / nc, hc = 64 * hpc;
    const int ar = nb * hpc < 4 ? nb * hpc : 4;
    P.nc = nc;
    P.stream_cta = dr_bytes(d, F, P.n_dec) / nc;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off += (bytes + 127) & ~(size_t)127;
        return (int)at;
    };
    auto max2 = [](size_t a, size_t b) { return a > b ? a : b; };
    P.cap = ((P.T > P.S ? P.T : P.S) + 15) & ~15;
    if (P.cap > ATT_CORE_MAX_KEYS || nc < 2 || dr_split(12 * hpc).tpw == 0 || dr_split(fc / 16).tpw == 0) return (size_t)-1;
    P.param_bytes = (int)((offsetof(DrParams, layer) + (size_t)P.n_dec * sizeof(DrLayer) + 15) & ~(size_t)15);
    take((size_t)P.param_bytes);
    P.stride_a = d + 64;  // 64 bytes past a multiple of 128: the eight rows of an
    P.stride_h = F + 64;  // operand load fall into distinct banks
    const size_t own = (size_t)((rb + nc - 1) / nc);
    P.off_bar = take(8 * (2 * DR_MAX_SLOTS + 2) + 8);
    P.off_a = take((size_t)rb * P.stride_a);
    P.off_h = take((size_t)rb * max2(P.stride_a, P.stride_h));
    P.off_y = take(own * d * 4);
    P.off_r = take(own * d * 4);
    P.off_q = take((size_t)rb * hc);
    P.off_red = take(max2((size_t)4 * 3 * nb * 512, (size_t)DR_WARPS * ar * P.cap * 4));
    P.off_stage = take(max2((size_t)rb * (hc + 4) * 4, max2((size_t)rb * (3 * hc + 16), (size_t)rb * (fc + 16))));
    P.off_prow = take((size_t)rb * P.cap);
    P.off_meta = take((size_t)(3 * rb + 8) * 4);
    // LayerNorm: the most warps per row (a power of two) that the owned rows
    // and the width leave
    int lw = 3;
    while (lw > 0 && ((int)own > (DR_WARPS >> lw) || d % (32 << lw) || d / (32 << lw) < 2 || (32 << lw) < d / 16)) lw--;
    P.ln_w = lw;
    P.ln_epl = d / (32 << lw);
    P.off_ln = take((size_t)DR_WARPS * (256 + d));
    P.off_ring = (int)off;
    if (off + 4 * DR_SLOT > max_smem) return (size_t)-1;
    int slots = (int)((max_smem - off) / DR_SLOT);
    P.slots = slots > DR_MAX_SLOTS ? DR_MAX_SLOTS : slots;
    int kd = 0;
    while (((d >> kd) & 1) == 0) kd++;
    P.ln_kd = kd;
    P.ln_dodd = d >> kd;
    P.ln_zm = P.ln_dodd > 1 ? ~0ull / (unsigned long long)P.ln_dodd : 0ull;  // floor(2^64 / ln_dodd)
    return off + (size_t)P.slots * DR_SLOT;
}

int dr_max_clusters(int nb, int hpc, int nc, size_t smem) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = dr_config(nc, 1, smem, nullptr, &attr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, dr_kernel(nb, hpc), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t decode_rows_init() {
    cudaError_t err = cudaSuccess;
    for (const auto &x : DR_FORMS)
        if (err == cudaSuccess)
            err = cudaFuncSetAttribute(dr_kernel(x[0], x[1]), cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    return err;
}

cudaError_t launch_decode_rows(const DrParams *dP, int nb, int hpc, int nc, int clusters, size_t smem, cudaStream_t st) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = dr_config(nc, clusters, smem, st, &attr);
    void *args[] = {(void *)&dP};
    return cudaLaunchKernelExC(&cfg, dr_kernel(nb, hpc), args);
}

}  // namespace mnmt
