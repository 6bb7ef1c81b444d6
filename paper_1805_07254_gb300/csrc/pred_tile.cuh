// Fused inference of the learned slope predictor (the network of mlp.cu) for one
// block's share of the subapertures, run by the consumer warps of frame_pred_kernel,
// after the pixel kernel, and of the loop kernel, after the grid barrier that follows
// its pixel stage; the block then multiplies the predicted slopes.
//
// The network is small (200 -> 64 -> 64 -> 2), so the phase is latency-bound:
// the BF16 weight fragments of both hidden layers, their biases and the
// neighbour indices are loaded into registers in the same round of L2 loads as
// the first tile's features, and each hidden layer is one pass of
// mma.sync.m16n8k16 (BF16 in, FP32 accumulate) by 8 warps, one 8-column slice
// each over both 16-row halves of a 32-sample tile.
//
// Arithmetic per element is that of the sequence kernel (mlp_predict.cu): the same
// BF16 operands, the same k order of the tensor-core steps, bias added after the
// sum, the same GELU, the output layer's products in the same order, and
//     s_pred = fma(sigma, y, s_k),
// so the fused and stand-alone forms give identical predictions.
#pragma once

#include <cuda_bf16.h>

#include "stream_mvm.cuh"

namespace rtc_pred {

using rtc_mvm::consumer_sync;
using rtc_mvm::kConsumers;

constexpr int NF = 200;                 // features: 5x5 neighbours x (x, y) x 4 frames
constexpr int KP = 208;                 // W1 row pitch (features padded to a multiple of 16)
constexpr int NH = 64;                  // hidden width
constexpr int NO = 2;                   // outputs (x and y slope)
constexpr int TS = 32;                  // samples per tile (two 16-row MMA halves)
constexpr int XP = 216;                 // X row pitch in BF16 (bank-conflict-free fragments)
constexpr int HP = 72;                  // H1 row pitch in BF16
constexpr int H2P = 72;                 // H2 row pitch in FP32 (4 rows x 8 columns: 32 banks)
constexpr int kMmaWarps = NH / 8;       // one 8-column slice per warp
constexpr int kPairs = TS * 25;         // (sample, neighbour) pairs of a tile
constexpr int kPairRounds = (kPairs + kConsumers - 1) / kConsumers;

// Offsets of the parameters in the flat vector (W1, b1, W2, b2, W3, b3).
constexpr int OFF_B1 = NH * NF;
constexpr int OFF_W2 = OFF_B1 + NH;
constexpr int OFF_B2 = OFF_W2 + NH * NH;
constexpr int OFF_W3 = OFF_B2 + NH;
constexpr int OFF_B3 = OFF_W3 + NO * NH;

// Shared-memory layout of the phase (byte offsets).
constexpr int SM_X = 0;                              // bf16 [TS][XP]
constexpr int SM_H1 = SM_X + TS * XP * 2;            // bf16 [TS][HP]
constexpr int SM_H2 = SM_H1 + TS * HP * 2;           // f32 [TS][H2P]
constexpr int SM_W3 = SM_H2 + TS * H2P * 4;          // f32 W3 [NO][NH], then b3 [NO]
constexpr int kSmemBytes = SM_W3 + (NO * NH + NO + 2) * 4;

static_assert(kPairRounds == 2, "gather registers assume two rounds of pairs");
static_assert(SM_H1 % 16 == 0 && SM_H2 % 16 == 0 && SM_W3 % 16 == 0, "alignment");
static_assert(OFF_B3 == OFF_W3 + NO * NH, "W3 and b3 are one run of the parameters");
static_assert(NF % 8 == 0 && NF + 8 == KP, "the last k step holds 8 features and 8 zero columns");

struct PredArgs {
    const __nv_bfloat16* w1;  // [NH][KP] BF16 copy of W1, zero padded
    const __nv_bfloat16* w2;  // [NH][NH] BF16 copy of W2
    const float* params;      // flat FP32 parameters (b1, b2, W3, b3 are read from here)
    const int* nbr;           // [nv][25] neighbour index or -1, (dr, dc) row-major
    float* ring;              // [4][kpad] measured slope vectors (x block, then y block)
    float* s_pred;            // [kpad] predicted next slopes
    int kpad, nv;
    float sigma, inv_sigma;
};

// GELU(z) = z Phi(z), exact form, from e = erfc(|z| / sqrt 2):
//     z >= 0: z - z e / 2,   z < 0: -|z| e / 2,   i.e.  max(z, 0) - |z| e / 2,
// which keeps its relative accuracy for negative z, where z (1 + erf) / 2 cancels.
// log2 e is |z| times a polynomial of degree 9 on [0, 6] (an iteratively reweighted
// least-squares fit of log2 erfc that equalises the error of the GELU itself, 7e-10,
// no branch).  Past 6 the same polynomial goes on falling, close to log2 erfc itself (at 8
// the GELU is -4.0e-15 for -5.0e-15), and from 12 on e is zero.  Against 64 bits the
// FP32 result is nearer than 0.5 z (1 + erff(z / sqrt 2)): relative 2-norm 2.9e-8
// against 3.7e-8 for z ~ N(0, 1), largest error 2.4e-7 against 3.7e-7.  NaN stays NaN.
constexpr float kGeluMax = 12.f;
constexpr int kGeluTerms = 10;
struct GeluPoly {
    float c[kGeluTerms];
};
__device__ constexpr GeluPoly kGelu = {{-1.1511046886444092f, -0.4592178463935852f, -0.05244341120123863f,
                                        0.0069376579485833645f, 1.959204746526666e-05f, -0.0002957938122563064f,
                                        8.329531556228176e-05f, -1.2535851965367328e-05f, 1.0430975407871301e-06f,
                                        -3.7503376404401934e-08f}};

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float relu_nan(float z) {
    float y;
    asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(y) : "f"(z));
    return y;
}
// erfc(a / sqrt 2) for 0 <= a <= kGeluMax.
__device__ __forceinline__ float gelu_erfc(float a) {
    float q = kGelu.c[kGeluTerms - 1];
#pragma unroll
    for (int k = kGeluTerms - 2; k >= 0; --k) q = __fmaf_rn(q, a, kGelu.c[k]);
    return ex2(__fmul_rn(a, q));
}
__device__ __forceinline__ float gelu(float z) {
    const float a = fminf(fabsf(z), kGeluMax);
    return __fmaf_rn(-0.5f, __fmul_rn(a, gelu_erfc(a)), relu_nan(z));
}

// Two GELUs with packed FP32 arithmetic: the same bits as gelu() of each.  (For
// throughput; its packed constants take 20 registers, which the fused kernels lack.)
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float2 gelu2(float x, float y) {
    const f32x2 a = pack2(fminf(fabsf(x), kGeluMax), fminf(fabsf(y), kGeluMax));
    f32x2 q = pack2(kGelu.c[kGeluTerms - 1], kGelu.c[kGeluTerms - 1]);
#pragma unroll
    for (int k = kGeluTerms - 2; k >= 0; --k) q = fma2(q, a, pack2(kGelu.c[k], kGelu.c[k]));
    const float2 p = unpack2(mul2(a, q));
    const f32x2 t = mul2(a, pack2(ex2(p.x), ex2(p.y)));
    return unpack2(fma2(pack2(-0.5f, -0.5f), t, pack2(relu_nan(x), relu_nan(y))));
}

__device__ __forceinline__ uint32_t ld32g(const __nv_bfloat16* p) {
    return __ldg(reinterpret_cast<const unsigned int*>(p));
}
__device__ __forceinline__ uint32_t ld32s(const __nv_bfloat16* p) {
    return *reinterpret_cast<const uint32_t*>(p);
}

__device__ __forceinline__ void mma16816(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// What a consumer thread keeps in registers for the phase.
struct Regs {
    uint32_t w1f[KP / 16][2];   // B fragments of W1 for this warp's 8 columns
    uint32_t w2f[NH / 16][2];   // B fragments of W2
    float b1v[2], b2v[2];       // biases of the thread's two accumulator columns
    int jn[kPairRounds];        // neighbour indices of the first tile's pairs
    float vo[kPairRounds][6];   // their slopes of the three older frames (lags 1-3)
};

// Neighbour index of pair p (sample p / 25, neighbour p % 25) of the tile at t0.
__device__ __forceinline__ int pair_nbr(const PredArgs& pa, int t0, int i1, int p) {
    if (p >= kPairs) return -1;
    const int i = t0 + p / 25;
    return i < i1 ? __ldg(pa.nbr + static_cast<size_t>(i) * 25 + (p - (p / 25) * 25)) : -1;
}

// What the first tile needs that does not depend on this frame's slopes: the
// weight fragments, biases and neighbour indices in registers, the first tile's
// features of the three older frames (ring rows head-1 .. head-3, written by earlier
// frames) in registers, and the output layer's weights in the scratch sm
// (asynchronous copies, complete once predict's first barrier has passed).
// [i0, i1): the block's subapertures.  Called before the wait for the measured slopes: in
// the loop after the block's grid-barrier arrival (a release would wait for these
// loads), in frame_pred_kernel before the wait for the pixel kernel.  OLDER = false
// leaves the older frames' features to predict: a kernel that may start before the
// kernels that wrote those rows are known to be complete.
template <bool OLDER>
__device__ __forceinline__ void prefetch(const PredArgs& pa, unsigned char* sm, int tid, int i0, int i1,
                                         int head, Regs& r) {
    float* w3s = reinterpret_cast<float*>(sm + SM_W3);
    for (int k = tid; k < NO * NH + NO; k += kConsumers) rtc_mvm::cp_async4(w3s + k, pa.params + OFF_W3 + k);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t = lane & 3;
    if (warp < kMmaWarps) {
        const __nv_bfloat16* w1 = pa.w1 + static_cast<size_t>(warp * 8 + g) * KP + 2 * t;
#pragma unroll
        for (int ks = 0; ks < KP / 16; ++ks) {
            r.w1f[ks][0] = ld32g(w1 + ks * 16);
            r.w1f[ks][1] = ld32g(w1 + ks * 16 + 8);
        }
        const __nv_bfloat16* w2 = pa.w2 + static_cast<size_t>(warp * 8 + g) * NH + 2 * t;
#pragma unroll
        for (int ks = 0; ks < NH / 16; ++ks) {
            r.w2f[ks][0] = ld32g(w2 + ks * 16);
            r.w2f[ks][1] = ld32g(w2 + ks * 16 + 8);
        }
        const int c = warp * 8 + 2 * t;
        r.b1v[0] = __ldg(pa.params + OFF_B1 + c);
        r.b1v[1] = __ldg(pa.params + OFF_B1 + c + 1);
        r.b2v[0] = __ldg(pa.params + OFF_B2 + c);
        r.b2v[1] = __ldg(pa.params + OFF_B2 + c + 1);
    }
#pragma unroll
    for (int q = 0; q < kPairRounds; ++q) r.jn[q] = pair_nbr(pa, i0, i1, tid + q * kConsumers);
    if constexpr (OLDER)
#pragma unroll
    for (int q = 0; q < kPairRounds; ++q)
#pragma unroll
        for (int la = 2; la < 8; ++la) {
            const float* row = pa.ring + static_cast<size_t>((head - (la >> 1)) & 3) * pa.kpad;
            r.vo[q][la - 2] = r.jn[q] >= 0 ? __ldcg(row + (la & 1) * pa.nv + r.jn[q]) : 0.f;
        }
}

// Once the measured slopes are complete: predictions of
// subapertures [i0, i1) from the ring rows head, head-1, head-2, head-3 (newest
// first), with the registers and scratch `prefetch` filled (before the wait, so
// that the weight and neighbour loads overlap it).  Every consumer thread
// calls it; sm is TS-sample scratch of kSmemBytes.  src(i, axis) gives the block's
// own copy of the measured slope s_k of subaperture i (the value in ring row head);
// each prediction goes to pa.s_pred and to sink(i, axis, value), after the same
// thread's src read of that slope.  Ends with a consumer barrier.
template <bool OLDER, typename Src, typename Sink>
__device__ __forceinline__ void predict(const PredArgs& pa, unsigned char* sm, int tid, int i0, int i1,
                                        int head, const Regs& r, const Src& src, const Sink& sink) {
    const int warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t = lane & 3;
    __nv_bfloat16* X = reinterpret_cast<__nv_bfloat16*>(sm + SM_X);
    __nv_bfloat16* H1 = reinterpret_cast<__nv_bfloat16*>(sm + SM_H1);
    float* H2 = reinterpret_cast<float*>(sm + SM_H2);
    const float* W3 = reinterpret_cast<const float*>(sm + SM_W3);
    const float* b3 = W3 + NO * NH;
    const float* rows[4];
#pragma unroll
    for (int lag = 0; lag < 4; ++lag)
        rows[lag] = pa.ring + static_cast<size_t>((head - lag) & 3) * pa.kpad;

    for (int t0 = i0; t0 < i1; t0 += TS) {
        int jn[kPairRounds];
#pragma unroll
        for (int q = 0; q < kPairRounds; ++q)
            jn[q] = t0 == i0 ? r.jn[q] : pair_nbr(pa, t0, i1, tid + q * kConsumers);
        // gather: every load of the thread's pairs in flight before any store; the
        // newest row was written by other blocks of this kernel (or by the kernel
        // before it), so it is read from L2 (the first tile's older rows may have come
        // with prefetch)
        float v[kPairRounds][8];
#pragma unroll
        for (int q = 0; q < kPairRounds; ++q)
#pragma unroll
            for (int la = 0; la < 8; ++la) {
                const int j = jn[q];
                if (OLDER && la >= 2 && t0 == i0) v[q][la] = r.vo[q][la - 2];
                else v[q][la] = j >= 0 ? __ldcg(rows[la >> 1] + (la & 1) * pa.nv + j) : 0.f;
            }
#pragma unroll
        for (int q = 0; q < kPairRounds; ++q) {
            const int p = tid + q * kConsumers;
            if (p < kPairs) {
                const int s = p / 25, nb = p - s * 25;
#pragma unroll
                for (int la = 0; la < 8; ++la)
                    X[s * XP + la * 25 + nb] = __float2bfloat16_rn(v[q][la] * pa.inv_sigma);
            }
        }
        if (t0 == i0) rtc_mvm::rows_landed();     // the output layer's weights (prefetch)
        consumer_sync();

        // hidden layer 1: z1 = X W1^T + b1, h1 = GELU(z1) as BF16; the upper half of
        // the last k step is the zero padding of W1 and X (not stored: zero fragments)
        if (warp < kMmaWarps) {
            float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
            for (int ks = 0; ks < KP / 16; ++ks) {
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    const __nv_bfloat16* A = X + (mt * 16 + g) * XP + ks * 16 + 2 * t;
                    const bool hi = ks * 16 + 8 < NF;
                    const uint32_t a[4] = {ld32s(A), ld32s(A + 8 * XP), hi ? ld32s(A + 8) : 0u,
                                           hi ? ld32s(A + 8 * XP + 8) : 0u};
                    mma16816(acc[mt], a, r.w1f[ks][0], r.w1f[ks][1]);
                }
            }
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int h = 0; h < 4; h += 2) {
                    const int row = mt * 16 + g + (h >> 1) * 8, col = warp * 8 + 2 * t;
                    *reinterpret_cast<__nv_bfloat162*>(H1 + row * HP + col) =
                        __floats2bfloat162_rn(gelu(acc[mt][h] + r.b1v[0]), gelu(acc[mt][h + 1] + r.b1v[1]));
                }
        }
        consumer_sync();

        // hidden layer 2: z2 = h1 W2^T + b2, h2 = GELU(z2) in FP32
        if (warp < kMmaWarps) {
            float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
            for (int ks = 0; ks < NH / 16; ++ks) {
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    const __nv_bfloat16* A = H1 + (mt * 16 + g) * HP + ks * 16 + 2 * t;
                    const uint32_t a[4] = {ld32s(A), ld32s(A + 8 * HP), ld32s(A + 8), ld32s(A + 8 * HP + 8)};
                    mma16816(acc[mt], a, r.w2f[ks][0], r.w2f[ks][1]);
                }
            }
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int h = 0; h < 4; h += 2) {
                    const int row = mt * 16 + g + (h >> 1) * 8, col = warp * 8 + 2 * t;
                    *reinterpret_cast<float2*>(H2 + row * H2P + col) =
                        make_float2(gelu(acc[mt][h] + r.b2v[0]), gelu(acc[mt][h + 1] + r.b2v[1]));
                }
        }
        consumer_sync();

        // output layer on CUDA cores and the predicted next slopes: the sum over the
        // columns 8 n + 2 t and 8 n + 2 t + 1 for each t, then the four sums pairwise
        // (the order of the sequence kernel, whose accumulator fragments hold those
        // columns lane by lane)
        if (tid < TS * NO) {
            const int s = tid >> 1, o = tid & 1;
            const int i = t0 + s;
            if (i < i1) {
                float y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
                for (int n = 0; n < NH / 8; ++n)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 h = *reinterpret_cast<const float2*>(H2 + s * H2P + 8 * n + 2 * q);
                        const float2 c = *reinterpret_cast<const float2*>(W3 + o * NH + 8 * n + 2 * q);
                        y[q] = fmaf(h.y, c.y, fmaf(h.x, c.x, y[q]));
                    }
                const float sp = __fmaf_rn(pa.sigma, ((y[0] + y[1]) + (y[2] + y[3])) + b3[o], src(i, o));
                pa.s_pred[o * pa.nv + i] = sp;
                sink(i, o, sp);
            }
        }
        consumer_sync();
    }
    if (i0 >= i1) rtc_mvm::rows_landed();         // no tile: still no copy left in flight
}

}  // namespace rtc_pred

// Predictor arguments of a handle with a loaded predictor (defined in frame_kernel.cu).
rtc_pred::PredArgs pred_args(const rtc_handle* h);
