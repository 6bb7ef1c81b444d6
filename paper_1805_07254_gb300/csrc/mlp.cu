// Learned slope predictor: a shared MLP 200 -> 64 -> 64 -> 2 with exact GELU,
// BF16 weights and activations in BF16 tensor-core GEMMs with FP32 accumulation.
//
// The paper has no learned component; this predictor offsets the one-frame servo
// lag of the integrator by predicting each subaperture's next slopes from the
// 5x5 neighbourhood of subapertures over the last 4 frames (200 features):
//   feature f = ((lag*2 + axis)*5 + (dr+2))*5 + (dc+2),   value / sigma
//   z1 = X W1^T + b1, h1 = GELU(z1), z2 = h1 W2^T + b2, h2 = GELU(z2),
//   y = h2 W3^T + b3,  next slopes = s_k + sigma * y.
// Training minimises sum((y - t)^2) / (2B) with t = (s_{k+1} - s_k) / sigma, by
// Adam with bias correction, on FP32 master weights.
//
// What bounds a training step.  4096 samples are 0.42 GFLOP (0.2 us of the chip's
// tensor peak): a step is a chain of dependent fetches (sample -> neighbour indices ->
// slopes), five small GEMMs and a reduction over the blocks.  So the tile is small, for
// every SM to get one (32 samples: 128 blocks at 4096), and nothing that is only used
// by the thread that made it goes through memory:
//   - one block of 8 warps takes 32 samples; warp w owns rows 16 (w & 1) and columns
//     16 (w >> 1) of z1, z2, dz2 and dz1 alike, so z, GELU' and h2 stay in its registers;
//   - the weights' B fragments go from L2 into registers while the features are fetched;
//   - X, h1, dz2 and dz1 lie in shared memory once, row by row; the weight-gradient
//     GEMMs, which contract over the samples, read them transposed by ldmatrix.trans;
//   - bias and W3 gradients are column sums in registers (shuffles, then the two row
//     halves);
//   - the 64 -> 2 layer and its gradient run on CUDA cores in FP32.
// A block runs several tiles when there are more than SMs, its weight gradients
// staying in the accumulators, and writes one partial vector; the update kernel sums
// the partials in a fixed order, applies Adam and refreshes the BF16 copies.  The two
// kernels overlap launch and drain (programmatic dependent launch); each waits for its
// predecessor before it touches memory that another kernel may write.
//
// Measured (ELT sequence, 4096 samples, step with update, GPU time): 13.0 us; 55 us with
// 64 blocks of 4 warps and 64 samples that kept z, transposed copies and column sums in
// shared memory between barriers, and one thread per parameter summing the partials.

#include <cuda_bf16.h>
#include <math.h>

#include "launch.cuh"
#include "mlp.h"
#include "pred_tile.cuh"
#include "rtc_internal.h"

namespace {

using rtc_pred::KP;
using rtc_pred::NF;
using rtc_pred::NH;
using rtc_pred::NO;
using rtc_pred::OFF_B1;
using rtc_pred::OFF_W2;
using rtc_pred::OFF_B2;
using rtc_pred::OFF_W3;
using rtc_pred::OFF_B3;
using rtc_pred::mma16816;
using rtc_mvm::smem_addr;

constexpr int OFF_W1 = 0;
constexpr int NPARAM = OFF_B3 + NO;
static_assert(NPARAM == RTC_MLP_NPARAMS, "parameter count");

constexpr int TM = kMlpTile;     // samples per tile
constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int XP = 216;          // row pitches in BF16: odd multiples of 16 bytes, so that
constexpr int HP = 72;           // the 8 rows of an ldmatrix tile fall in different banks
constexpr int kSteps1 = KP / 16, kSteps2 = NH / 16, kStepsB = TM / 16;
constexpr int kN1 = KP / 16;     // 8-column tiles of dW1 a warp owns (half of KP / 8)
static_assert(TM == 32 && kMlpPartPitch % 64 == 0 && kMlpPartPitch > NPARAM, "tile and pitch");

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}
__device__ __forceinline__ void ldsm2t(uint32_t (&r)[2], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}

// GELU(z) and its derivative Phi(z) + z phi(z); the same e as rtc_pred::gelu.
__device__ __forceinline__ float2 gelu_both(float z) {
    const float a = fminf(fabsf(z), rtc_pred::kGeluMax);
    const float e = rtc_pred::gelu_erfc(a);
    const float cdf = z >= 0.f ? __fmaf_rn(-0.5f, e, 1.f) : 0.5f * e;
    const float pdf = 0.39894228040143268f * rtc_pred::ex2(-0.72134752044448170f * z * z);
    return make_float2(__fmaf_rn(-0.5f, __fmul_rn(a, e), rtc_pred::relu_nan(z)), __fmaf_rn(z, pdf, cdf));
}

struct Smem {
    alignas(16) bf16 X[TM * XP];      // features
    alignas(16) bf16 H1[TM * HP];     // first hidden activation
    alignas(16) bf16 DZ2[TM * HP];    // back-propagated dz2, dz1
    alignas(16) bf16 DZ1[TM * HP];
    alignas(16) bf16 W2[NH * HP];     // W2 [n][k], for dh1 = dz2 W2
    float w3[NO * NH + NO];           // W3, b3
    float b1[NH], b2[NH];
    float yp[4][TM][NO];              // output sums of the four column quarters
    float tgt[TM][NO];
    float col[2][4][NH];              // column sums of the row halves: db2, dW3[0], dW3[1], db1
    float red[2][3];                  // loss and db3 of the row halves
};

// What a thread keeps over the tiles of its block.
struct Weights {
    uint32_t w1[kSteps1][2][2];       // B fragments of the warp's 16 columns
    uint32_t w2[kSteps2][2][2];
};
struct Grads {
    float w1[kN1][4];                 // dW1: rows 16 (w & 3), columns 104 (w >> 2)
    float w2[4][4];                   // dW2: rows 16 (w & 3), columns 32 (w >> 2)
    float bias[2];                    // the thread's column sum (db2, dW3, db1) and loss or db3
};

__device__ __forceinline__ void load_weights(Smem& sm, const MlpDev& w, Weights& r) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t = lane & 3, n0 = (warp >> 1) * 16;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
        const bf16* p1 = w.w1_bf16 + static_cast<size_t>(n0 + nt * 8 + g) * KP + 2 * t;
#pragma unroll
        for (int ks = 0; ks < kSteps1; ++ks) {
            r.w1[ks][nt][0] = *reinterpret_cast<const uint32_t*>(p1 + ks * 16);
            r.w1[ks][nt][1] = *reinterpret_cast<const uint32_t*>(p1 + ks * 16 + 8);
        }
        const bf16* p2 = w.w2_bf16 + static_cast<size_t>(n0 + nt * 8 + g) * NH + 2 * t;
#pragma unroll
        for (int ks = 0; ks < kSteps2; ++ks) {
            r.w2[ks][nt][0] = *reinterpret_cast<const uint32_t*>(p2 + ks * 16);
            r.w2[ks][nt][1] = *reinterpret_cast<const uint32_t*>(p2 + ks * 16 + 8);
        }
    }
    for (int i = tid; i < NH * NH / 8; i += kThreads) {
        const int n = i / (NH / 8), c = i - n * (NH / 8);
        *reinterpret_cast<uint4*>(sm.W2 + n * HP + 8 * c) = reinterpret_cast<const uint4*>(w.w2_bf16)[i];
    }
    for (int i = tid; i < NO * NH + NO; i += kThreads) sm.w3[i] = w.master[OFF_W3 + i];
    if (tid < NH) sm.b1[tid] = w.master[OFF_B1 + tid];
    else if (tid < 2 * NH) sm.b2[tid - NH] = w.master[OFF_B2 + tid - NH];
}

// X's padding columns (zero weights meet them: they must be finite).
__device__ __forceinline__ void clear_padding(Smem& sm) {
    for (int q = threadIdx.x; q < TM * (XP - NF); q += kThreads)
        sm.X[(q / (XP - NF)) * XP + NF + q % (XP - NF)] = __float2bfloat16_rn(0.f);
}

// Features of an explicit batch X [B][NF]; rows past B are zero.
__device__ __forceinline__ void fill_rows(Smem& sm, const float* __restrict__ X, int s0, int ns) {
    constexpr int kPer = TM * NF / kThreads;             // 25 values a thread, all in flight
    static_assert(TM * NF % kThreads == 0, "even split");
    float v[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int q = threadIdx.x + j * kThreads;
        v[j] = q < ns * NF ? __ldcg(X + static_cast<size_t>(s0) * NF + q) : 0.f;
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int q = threadIdx.x + j * kThreads, s = q / NF;
        sm.X[s * XP + q - s * NF] = __float2bfloat16_rn(v[j]);
    }
}

// Features and targets of samples (subaperture, frame k) of a slope sequence S: frames
// k .. k-3 and (S[k+1] - S[k]) / sigma.  A sample outside the sequence or the pupil
// contributes zeros.  By (sample, neighbour) pairs, every load of a round in flight.
struct Seq {
    const float* S;
    const int* nbr;
    const int2* samples;
    int n_frames, nv;
    float inv_sigma;
};
__device__ __forceinline__ void fill_seq(Smem& sm, const Seq& q, int s0, int ns) {
    const size_t row = 2 * static_cast<size_t>(q.nv);
    const int tid = threadIdx.x;
    auto sample = [&](int s) {
        int2 sk = s < ns ? q.samples[s0 + s] : make_int2(-1, 0);
        if (!(sk.x >= 0 && sk.x < q.nv && sk.y >= 3 && sk.y <= q.n_frames - 2)) sk.x = -1;
        return sk;
    };
    constexpr int kPairs = TM * 25, kRounds = (kPairs + kThreads - 1) / kThreads;
    int2 sk[kRounds];
    int j[kRounds];
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        const int p = tid + r * kThreads;
        sk[r] = p < kPairs ? sample(p / 25) : make_int2(-1, 0);
    }
    // the targets' samples: one more round for the first two warps
    const int2 st = tid < TM * NO ? sample(tid >> 1) : make_int2(-1, 0);
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        const int p = tid + r * kThreads;
        j[r] = sk[r].x >= 0 ? __ldg(q.nbr + static_cast<size_t>(sk[r].x) * 25 + p % 25) : -1;
    }
    float t0 = 0.f, t1 = 0.f;
    if (st.x >= 0) {
        const float* p = q.S + st.y * row + (tid & 1) * q.nv + st.x;
        t0 = p[0];
        t1 = p[row];
    }
#pragma unroll
    for (int r0 = 0; r0 < kRounds; r0 += 2) {
        float v[2][8];
#pragma unroll
        for (int d = 0; d < 2; ++d)
#pragma unroll
            for (int la = 0; la < 8; ++la) {
                const int r = r0 + d;
                v[d][la] = j[r] >= 0 ? q.S[(sk[r].y - (la >> 1)) * row + (la & 1) * q.nv + j[r]] : 0.f;
            }
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            const int p = tid + (r0 + d) * kThreads;
            if (p < kPairs) {
                bf16* x = sm.X + (p / 25) * XP + p % 25;
#pragma unroll
                for (int la = 0; la < 8; ++la) x[la * 25] = __float2bfloat16_rn(v[d][la] * q.inv_sigma);
            }
        }
    }
    if (tid < TM * NO) sm.tgt[tid >> 1][tid & 1] = (t1 - t0) * q.inv_sigma;
    static_assert(kRounds % 2 == 0, "rounds go in pairs");
}

// Shared-memory address of the thread's row of an ldmatrix.x4 over a 16x16 tile at
// (r0, c0) of a [..][ld] BF16 array.  Not transposed: A fragments (rows = samples).
// Read by ldmatrix.trans, tile_row gives B fragments (rows = k, columns = n) and
// tile_row_t A fragments of the transpose (rows = k, columns = m).
__device__ __forceinline__ uint32_t tile_row(const bf16* base, int ld, int r0, int c0) {
    const int l = threadIdx.x & 31;
    return smem_addr(base + (r0 + (l & 15)) * ld + c0 + (l >> 4) * 8);
}
__device__ __forceinline__ uint32_t tile_row_t(const bf16* base, int ld, int r0, int c0) {
    const int l = threadIdx.x & 31;
    return smem_addr(base + (r0 + (l & 7) + (l >> 4) * 8) * ld + c0 + ((l >> 3) & 1) * 8);
}

// Sum over the 16 rows of the warp's half: v holds the thread's two rows added.
__device__ __forceinline__ float rows_sum(float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    return v + __shfl_xor_sync(0xffffffffu, v, 16);
}

struct Hidden {
    float g1[2][4], g2[2][4], h2[2][4];   // GELU'(z1), GELU'(z2), h2 of the warp's fragment
};

// Forward pass of the tile in sm.X; leaves the column quarters' output sums in sm.yp
// (complete after the closing barrier).
template <bool GRAD>
__device__ __forceinline__ void forward_tile(Smem& sm, const Weights& w, Hidden& hd) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int m0 = (warp & 1) * 16, n0 = (warp >> 1) * 16;
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int ks = 0; ks < kSteps1; ++ks) {
        uint32_t a[4];
        ldsm4(a, tile_row(sm.X, XP, m0, ks * 16));
        mma16816(acc[0], a, w.w1[ks][0][0], w.w1[ks][0][1]);
        mma16816(acc[1], a, w.w1[ks][1][0], w.w1[ks][1][1]);
    }
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int h = 0; h < 4; h += 2) {
            const int r = m0 + g + h * 4, c = n0 + nt * 8 + 2 * t;
            const float z0 = acc[nt][h] + sm.b1[c], z1 = acc[nt][h + 1] + sm.b1[c + 1];
            float2 v;
            if (GRAD) {
                const float2 p = gelu_both(z0), q = gelu_both(z1);
                v = make_float2(p.x, q.x);
                hd.g1[nt][h] = p.y;
                hd.g1[nt][h + 1] = q.y;
            } else {
                v = rtc_pred::gelu2(z0, z1);
            }
            *reinterpret_cast<__nv_bfloat162*>(sm.H1 + r * HP + c) = __floats2bfloat162_rn(v.x, v.y);
            acc[nt][h] = acc[nt][h + 1] = 0.f;
        }
    __syncthreads();
#pragma unroll
    for (int ks = 0; ks < kSteps2; ++ks) {
        uint32_t a[4];
        ldsm4(a, tile_row(sm.H1, HP, m0, ks * 16));
        mma16816(acc[0], a, w.w2[ks][0][0], w.w2[ks][0][1]);
        mma16816(acc[1], a, w.w2[ks][1][0], w.w2[ks][1][1]);
    }
    float y[2][NO] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int c = n0 + nt * 8 + 2 * t + (h & 1);
            const float z = acc[nt][h] + sm.b2[c];
            const float2 p = GRAD ? gelu_both(z) : make_float2(rtc_pred::gelu(z), 0.f);
            hd.h2[nt][h] = p.x;
            hd.g2[nt][h] = p.y;
#pragma unroll
            for (int o = 0; o < NO; ++o) y[h >> 1][o] = fmaf(p.x, sm.w3[o * NH + c], y[h >> 1][o]);
        }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int o = 0; o < NO; ++o) {
            float v = y[r][o];
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            if (t == 0) sm.yp[warp >> 1][m0 + g + 8 * r][o] = v;
        }
    __syncthreads();
}

// Output of row s: the quarters pairwise, then b3.
__device__ __forceinline__ float output(const Smem& sm, int s, int o) {
    return (sm.yp[0][s][o] + sm.yp[1][s][o]) + (sm.yp[2][s][o] + sm.yp[3][s][o]) + sm.w3[NO * NH + o];
}

// Backward pass of the tile; adds to gr and, on the threads that own them, to the
// running bias, W3 and loss sums.
__device__ __forceinline__ void backward_tile(Smem& sm, const Hidden& hd, int ns, float inv_batch, Grads& gr) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t = lane & 3;
    const int m0 = (warp & 1) * 16, n0 = (warp >> 1) * 16;
    float e[2][NO], dy[2][NO];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int o = 0; o < NO; ++o) {
            const int s = m0 + g + 8 * r;
            e[r][o] = s < ns ? output(sm, s, o) - sm.tgt[s][o] : 0.f;
            dy[r][o] = e[r][o] * inv_batch;
        }
    if (warp < 2) {                                        // loss and db3 of the row half
        const float l = rows_sum(fmaf(e[0][0], e[0][0], e[0][1] * e[0][1]) + fmaf(e[1][0], e[1][0], e[1][1] * e[1][1]));
        const float d0 = rows_sum(dy[0][0] + dy[1][0]), d1 = rows_sum(dy[0][1] + dy[1][1]);
        if (lane == 0) {
            sm.red[warp][0] = l;
            sm.red[warp][1] = d0;
            sm.red[warp][2] = d1;
        }
    }
    // dz2 = (dy W3) GELU'(z2), as BF16 for the GEMMs; db2 and dW3 from the FP32 values
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
        const int c = n0 + nt * 8 + 2 * t;
        float dz[4];
#pragma unroll
        for (int h = 0; h < 4; ++h)
            dz[h] = fmaf(dy[h >> 1][1], sm.w3[NH + c + (h & 1)], dy[h >> 1][0] * sm.w3[c + (h & 1)]) * hd.g2[nt][h];
#pragma unroll
        for (int r = 0; r < 2; ++r)
            *reinterpret_cast<__nv_bfloat162*>(sm.DZ2 + (m0 + g + 8 * r) * HP + c) =
                __floats2bfloat162_rn(dz[2 * r], dz[2 * r + 1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float b = rows_sum(dz[h] + dz[2 + h]);
            const float a0 = rows_sum(fmaf(dy[0][0], hd.h2[nt][h], dy[1][0] * hd.h2[nt][2 + h]));
            const float a1 = rows_sum(fmaf(dy[0][1], hd.h2[nt][h], dy[1][1] * hd.h2[nt][2 + h]));
            if (g == 0) {
                sm.col[warp & 1][0][c + h] = b;
                sm.col[warp & 1][1][c + h] = a0;
                sm.col[warp & 1][2][c + h] = a1;
            }
        }
    }
    __syncthreads();
    // dh1 = dz2 W2, dz1 = dh1 GELU'(z1)
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int ks = 0; ks < kSteps2; ++ks) {
        uint32_t a[4], b[4];
        ldsm4(a, tile_row(sm.DZ2, HP, m0, ks * 16));
        ldsm4t(b, tile_row(sm.W2, HP, ks * 16, n0));
        mma16816(acc[0], a, b[0], b[1]);
        mma16816(acc[1], a, b[2], b[3]);
    }
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
        const int c = n0 + nt * 8 + 2 * t;
#pragma unroll
        for (int h = 0; h < 4; ++h) acc[nt][h] *= hd.g1[nt][h];
#pragma unroll
        for (int r = 0; r < 2; ++r)
            *reinterpret_cast<__nv_bfloat162*>(sm.DZ1 + (m0 + g + 8 * r) * HP + c) =
                __floats2bfloat162_rn(acc[nt][2 * r], acc[nt][2 * r + 1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float b = rows_sum(acc[nt][h] + acc[nt][2 + h]);
            if (g == 0) sm.col[warp & 1][3][c + h] = b;
        }
    }
    // dW2 = dz2^T h1
    const int mr = (warp & 3) * 16, nh = warp >> 2;
#pragma unroll
    for (int ks = 0; ks < kStepsB; ++ks) {
        uint32_t a[4], b[4];
        ldsm4t(a, tile_row_t(sm.DZ2, HP, ks * 16, mr));
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            ldsm4t(b, tile_row(sm.H1, HP, ks * 16, nh * 32 + p * 16));
            mma16816(gr.w2[2 * p], a, b[0], b[1]);
            mma16816(gr.w2[2 * p + 1], a, b[2], b[3]);
        }
    }
    __syncthreads();
    // dW1 = dz1^T X
#pragma unroll
    for (int ks = 0; ks < kStepsB; ++ks) {
        uint32_t a[4];
        ldsm4t(a, tile_row_t(sm.DZ1, HP, ks * 16, mr));
#pragma unroll
        for (int p = 0; p < kN1 / 2; ++p) {
            uint32_t b[4];
            ldsm4t(b, tile_row(sm.X, XP, ks * 16, nh * kN1 * 8 + p * 16));
            mma16816(gr.w1[2 * p], a, b[0], b[1]);
            mma16816(gr.w1[2 * p + 1], a, b[2], b[3]);
        }
        uint32_t b[2];
        ldsm2t(b, tile_row(sm.X, XP, ks * 16, nh * kN1 * 8 + (kN1 - 1) * 8));
        mma16816(gr.w1[kN1 - 1], a, b[0], b[1]);
    }
    // the tile's column sums: thread c the bias columns, three threads the rest
    if (tid < 4 * NH) gr.bias[0] += sm.col[0][tid >> 6][tid & 63] + sm.col[1][tid >> 6][tid & 63];
    if (tid < 3) gr.bias[1] += sm.red[0][tid] + sm.red[1][tid];
}

// The block's partial gradient (and loss sum, last).
__device__ __forceinline__ void write_part(const Grads& gr, float* __restrict__ part) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t = lane & 3, mr = (warp & 3) * 16, nh = warp >> 2;
#pragma unroll
    for (int nt = 0; nt < kN1; ++nt) {
        const int c = (nh * kN1 + nt) * 8 + 2 * t;
        if (c < NF)
#pragma unroll
            for (int r = 0; r < 2; ++r)
                *reinterpret_cast<float2*>(part + OFF_W1 + (mr + g + 8 * r) * NF + c) =
                    make_float2(gr.w1[nt][2 * r], gr.w1[nt][2 * r + 1]);
    }
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int r = 0; r < 2; ++r)
            *reinterpret_cast<float2*>(part + OFF_W2 + (mr + g + 8 * r) * NH + nh * 32 + nt * 8 + 2 * t) =
                make_float2(gr.w2[nt][2 * r], gr.w2[nt][2 * r + 1]);
    // col: db2, dW3[0], dW3[1], db1; red: loss, db3[0], db3[1]
    const int k = tid >> 6, c = tid & 63;
    part[(k == 0 ? OFF_B2 : k == 3 ? OFF_B1 : OFF_W3 + (k - 1) * NH) + c] = gr.bias[0];
    if (tid < 3) part[tid == 0 ? NPARAM : OFF_B3 + tid - 1] = gr.bias[1];
}

// ---- kernels --------------------------------------------------------------------

template <typename Fill>
__device__ __forceinline__ void train_body(Smem& sm, const MlpDev& w, int B, float* __restrict__ parts,
                                           const Fill& fill) {
    // the weights are the previous update's and the inputs may be any earlier kernel's
    pdl_wait();
    pdl_launch_dependents();
    Weights wr;
    Grads gr;
#pragma unroll
    for (int i = 0; i < kN1; ++i) gr.w1[i][0] = gr.w1[i][1] = gr.w1[i][2] = gr.w1[i][3] = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) gr.w2[i][0] = gr.w2[i][1] = gr.w2[i][2] = gr.w2[i][3] = 0.f;
    gr.bias[0] = gr.bias[1] = 0.f;
    load_weights(sm, w, wr);
    clear_padding(sm);
    const float inv_batch = 1.f / static_cast<float>(B);
    for (int tile = blockIdx.x, tiles = mlp_tiles(B); tile < tiles; tile += gridDim.x) {
        const int s0 = tile * TM, ns = min(TM, B - s0);
        if (tile >= static_cast<int>(gridDim.x)) __syncthreads();         // the last tile's reads of X
        fill(s0, ns);
        __syncthreads();
        Hidden hd;
        forward_tile<true>(sm, wr, hd);
        backward_tile(sm, hd, ns, inv_batch, gr);
    }
    write_part(gr, parts + static_cast<size_t>(blockIdx.x) * kMlpPartPitch);
}

// Explicit batch: X [B][NF] FP32 (row-major), targets T [B][NO].
__global__ void __launch_bounds__(kThreads, 1) mlp_train_kernel(MlpDev w, const float* __restrict__ X,
                                                                const float* __restrict__ T, int B,
                                                                float* __restrict__ parts) {
    __shared__ Smem sm;
    train_body(sm, w, B, parts, [&](int s0, int ns) {
        fill_rows(sm, X, s0, ns);
        for (int i = threadIdx.x; i < TM * NO; i += kThreads)
            sm.tgt[i / NO][i % NO] = i / NO < ns ? __ldcg(T + static_cast<size_t>(s0) * NO + i) : 0.f;
    });
}

__global__ void __launch_bounds__(kThreads, 1) mlp_train_seq_kernel(MlpDev w, Seq q, int B, float* __restrict__ parts) {
    __shared__ Smem sm;
    train_body(sm, w, B, parts, [&](int s0, int ns) { fill_seq(sm, q, s0, ns); });
}

__global__ void __launch_bounds__(kThreads, 1) mlp_forward_kernel(MlpDev w, const float* __restrict__ X, int B,
                                                                  float* __restrict__ Yout) {
    __shared__ Smem sm;
    Weights wr;
    load_weights(sm, w, wr);
    clear_padding(sm);
    for (int tile = blockIdx.x, tiles = mlp_tiles(B); tile < tiles; tile += gridDim.x) {
        const int s0 = tile * TM, ns = min(TM, B - s0);
        fill_rows(sm, X, s0, ns);
        __syncthreads();
        Hidden hd;
        forward_tile<false>(sm, wr, hd);
        for (int i = threadIdx.x; i < ns * NO; i += kThreads)
            Yout[static_cast<size_t>(s0) * NO + i] = output(sm, i / NO, i % NO);
    }
}

// Sum of the block partials, then (when lr > 0) one Adam step on the FP32 master weights
// and a refresh of the BF16 copies.  A block takes 64 parameters: 16 lanes of float4 by
// 16 groups of partials (group q adds the partials q, q + 16, ... in turn), then the 16
// sums pairwise.  grad_out (optional) receives the summed gradient; loss_out (optional)
// the loss sum / (2B).
constexpr int kUpdateParams = 64;
__global__ void __launch_bounds__(256) mlp_update_kernel(MlpDev w, const float* __restrict__ parts, int nparts,
                                                         float inv_2b, float lr, float beta1, float beta2, float eps,
                                                         float bc1, float bc2, float* __restrict__ grad_out,
                                                         float* __restrict__ loss_out) {
    __shared__ float4 red[16][17];
    const int tid = threadIdx.x, lane = tid & 15, grp = tid >> 4;
    const int p = blockIdx.x * kUpdateParams + tid;
    // the step's own state: last written by the update before the train kernel that
    // this launch depends on, which waited for it before it let this one start
    const bool own = tid < kUpdateParams && p < NPARAM && lr > 0.f;
    const float m0 = own ? __ldcg(w.m + p) : 0.f, v0 = own ? __ldcg(w.v + p) : 0.f;   // (never from a stale L1)
    const float w0 = own ? __ldcg(w.master + p) : 0.f;
    pdl_wait();
    pdl_launch_dependents();
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4* src = reinterpret_cast<const float4*>(parts + blockIdx.x * kUpdateParams) + lane;
    for (int c0 = grp; c0 < nparts; c0 += 16 * 8) {
        float4 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            v[i] = c0 + 16 * i < nparts ? __ldcg(src + static_cast<size_t>(c0 + 16 * i) * (kMlpPartPitch / 4))
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            s.x += v[i].x;
            s.y += v[i].y;
            s.z += v[i].z;
            s.w += v[i].w;
        }
    }
    red[grp][lane] = s;
    __syncthreads();
    if (tid >= kUpdateParams || p > NPARAM) return;
    float t[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) t[q] = reinterpret_cast<const float*>(&red[q][0])[tid];
#pragma unroll
    for (int width = 1; width < 16; width <<= 1)
#pragma unroll
        for (int q = 0; q < 16; q += 2 * width) t[q] += t[q + width];
    const float g = t[0];
    if (p == NPARAM) {
        if (loss_out) *loss_out = g * inv_2b;
        return;
    }
    if (grad_out) grad_out[p] = g;
    if (lr > 0.f) {
        const float m = beta1 * m0 + (1.f - beta1) * g;
        const float v = beta2 * v0 + (1.f - beta2) * g * g;
        w.m[p] = m;
        w.v[p] = v;
        const float mh = m / bc1, vh = v / bc2;
        const float np = w0 - lr * mh / (sqrtf(vh) + eps);
        w.master[p] = np;
        if (p < OFF_B1) {
            const int r = p / NF, c = p - r * NF;
            w.w1_bf16[r * KP + c] = __float2bfloat16_rn(np);
        } else if (p >= OFF_W2 && p < OFF_B2) {
            w.w2_bf16[p - OFF_W2] = __float2bfloat16_rn(np);
        }
    }
}

__global__ void mlp_refresh_kernel(MlpDev w) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < NH * KP) {
        const int r = p / KP, c = p - r * KP;
        w.w1_bf16[p] = __float2bfloat16_rn(c < NF ? w.master[OFF_W1 + r * NF + c] : 0.f);
    }
    if (p < NH * NH) w.w2_bf16[p] = __float2bfloat16_rn(w.master[OFF_W2 + p]);
}

}  // namespace

cudaError_t mlp_launch_refresh(const MlpDev& w, cudaStream_t st) {
    mlp_refresh_kernel<<<(NH * KP + 255) / 256, 256, 0, st>>>(w);
    return cudaGetLastError();
}

cudaError_t mlp_launch_train(const MlpDev& w, const float* X, const float* T, int B, float* parts, int blocks,
                             cudaStream_t st) {
    return launch_pdl(mlp_train_kernel, dim3(blocks), dim3(kThreads), 0, st, w, X, T, B, parts);
}

cudaError_t mlp_launch_train_seq(const MlpDev& w, const float* S, int n_frames, int nv, const int* nbr,
                                 const int2* samples, int B, float inv_sigma, float* parts, int blocks,
                                 cudaStream_t st) {
    const Seq q{S, nbr, samples, n_frames, nv, inv_sigma};
    return launch_pdl(mlp_train_seq_kernel, dim3(blocks), dim3(kThreads), 0, st, w, q, B, parts);
}

cudaError_t mlp_launch_forward(const MlpDev& w, const float* X, int B, float* Y, int sms, cudaStream_t st) {
    mlp_forward_kernel<<<mlp_blocks(B, sms), kThreads, 0, st>>>(w, X, B, Y);
    return cudaGetLastError();
}

cudaError_t mlp_launch_update(const MlpDev& w, const float* parts, int nparts, int B, float lr,
                              float beta1, float beta2, float eps, int step, float* grad_out,
                              float* loss_out, cudaStream_t st) {
    const float bc1 = 1.f - powf(beta1, static_cast<float>(step));
    const float bc2 = 1.f - powf(beta2, static_cast<float>(step));
    return launch_pdl(mlp_update_kernel, dim3(kMlpPartPitch / kUpdateParams), dim3(256), 0, st, w, parts, nparts,
                      0.5f / B, lr, beta1, beta2, eps, bc1, bc2, grad_out, loss_out);
}
