// The slope predictor over a recorded sequence (rtc_mlp_predict_seq): every frame and
// every subaperture in one launch.
//
// What bounds it.  A prediction is 2 x (200x64 + 64x64 + 128) operations on 200
// features, 16 bytes of new slopes: arithmetic, not memory.  Per 32 samples a warp
// issues 272 mma.sync, 2 x 2,048 GELUs (the larger half of its instructions) and the
// shared-memory reads of its fragments.  The products stay on mma.sync.m16n8k16: a
// sequence scored offline equals the prediction fused into the frame kernel
// (pred_tile.cuh) bit for bit, so both take the same instruction in the same k order.
//
// Split.  A warp takes 32 samples (consecutive subapertures) and runs them through
// consecutive frames on its own: no block barrier after the weights are loaded.
//   - Features slide: of a sample's 200 features 150 are those of the frame before.
//     The warp keeps a ring of 4 frames of BF16 features in shared memory and gathers
//     only the newest frame's 50 per sample, a lane per sample (neighbouring lanes read
//     neighbouring slopes), the next frame's loads issued ahead of the products.
//   - Layer 1 accumulators are the layout that layer 2 wants as its A fragments, so the
//     hidden activations never leave registers; the 64 -> 2 layer is 16 products a lane
//     and two shuffles.
//   - The weights lie in shared memory in fragment order, one 16-byte read per lane for
//     two 8-column tiles, each read serving both 16-row halves.
// The units (32 samples x 1 frame) are dealt to the warps in contiguous runs, tile by
// tile, so a warp refills its ring (3 older frames) once or twice.
//
// Measured (ELT, 3,972 subapertures x 996 frames, 135 GFLOP): 0.55 ms; one launch per
// frame of 64-sample blocks, each loading the weights and gathering all 200 features
// again, took 18.4 ms.  mma.sync is issued in 0.22 ms of that (1,024 multiply-adds a
// clock and SM); products and GELUs of the two warps of a scheduler overlap only in
// part.  12 warps of 168 registers came to 0.56 ms, 13 of 128 to 0.67.

#include <cuda_bf16.h>

#include <algorithm>

#include "mlp.h"
#include "pred_tile.cuh"
#include "rtc_internal.h"

namespace {

using rtc_pred::KP;
using rtc_pred::mma16816;
using rtc_pred::NH;
using rtc_pred::NO;
using rtc_pred::OFF_B1;
using rtc_pred::OFF_B2;
using rtc_pred::OFF_W3;

constexpr int kMaxWarps = 8;             // 255 registers a thread (see above)
constexpr int kTile = 32;                // samples a warp takes at a time
constexpr int kLagWords = 25;            // BF16 pairs of one frame's 50 features
constexpr int kPitch = 28;               // words per sample and frame: 4 x 7, so that the 8
                                         // rows x 4 words of a fragment load are 32 banks
constexpr int kSlot = kTile * kPitch * 4;            // bytes of one frame of a warp's ring
constexpr int kSteps1 = KP / 16, kSteps2 = NH / 16;  // k steps of the two layers

// Shared memory: weights in fragment order, then the rings.
constexpr int SW1 = 0;                                // uint4 [13][4][32]
constexpr int SW2 = SW1 + kSteps1 * 4 * 32 * 16;      // uint4 [4][4][32]
constexpr int SB1 = SW2 + kSteps2 * 4 * 32 * 16;      // f32 [64]
constexpr int SB2 = SB1 + NH * 4;                     // f32 [64]
constexpr int SW3 = SB2 + NH * 4;                     // f32 [2][64], b3 [2], pad
constexpr int SRING = SW3 + (NO * NH + 4) * 4;
constexpr int smem_bytes(int warps) { return SRING + warps * 4 * kSlot; }
static_assert(SRING % 16 == 0 && kSlot % 16 == 0, "alignment");
static_assert(smem_bytes(kMaxWarps) <= 227 * 1024, "shared memory");

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// One axis (25 neighbours) of one frame for the lane's sample: off[nb] is the byte
// offset of the neighbour's slope in the axis block, or ~0 off the pupil.
__device__ __forceinline__ void load_axis(const float* __restrict__ row, const unsigned (&off)[25], float (&v)[25]) {
#pragma unroll
    for (int nb = 0; nb < 25; ++nb)
        v[nb] = off[nb] != ~0u ? __ldg(reinterpret_cast<const float*>(reinterpret_cast<const char*>(row) + off[nb]))
                               : 0.f;
}

// The x features (words 0 .. 11; x of neighbour 24 shares word 12 with the first y) and
// the y features of the lane's sample into its row of a ring slot.
__device__ __forceinline__ uint32_t store_x(unsigned char* dst, const float (&v)[25], float inv_sigma) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            w[j] = pack_bf16(v[8 * q + 2 * j] * inv_sigma, v[8 * q + 2 * j + 1] * inv_sigma);
        reinterpret_cast<uint4*>(dst)[q] = make_uint4(w[0], w[1], w[2], w[3]);
    }
    return pack_bf16(v[24] * inv_sigma, 0.f);
}
__device__ __forceinline__ void store_y(unsigned char* dst, const float (&v)[25], float inv_sigma, uint32_t x24) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int f = 8 * q + 2 * j - 1;          // y neighbours f and f + 1 (word 12 + 4 q + j)
            const float lo = f >= 0 && f < 25 ? v[f < 0 ? 0 : f > 24 ? 24 : f] * inv_sigma : 0.f;
            const float hi = f + 1 < 25 ? v[f + 1 > 24 ? 24 : f + 1] * inv_sigma : 0.f;
            w[j] = pack_bf16(lo, hi);
        }
        if (q == 0) w[0] = (w[0] & 0xffff0000u) | (x24 & 0xffffu);
        reinterpret_cast<uint4*>(dst + 48)[q] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

__global__ void __launch_bounds__(kMaxWarps * 32, 1)
mlp_predict_seq_kernel(MlpDev w, const float* __restrict__ S, float* __restrict__ out, int k0, int nk, int nv,
                       const int* __restrict__ nbr, float sigma, int tiles) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t = lane & 3;
    // weights: fragment (ks, column tiles 2p and 2p + 1) of a lane is one uint4
    auto frag = [&](const __nv_bfloat16* W, int ld, int i) {
        const int l = i & 31, p = (i >> 5) & 3, ks = i >> 7;
        const __nv_bfloat16* b = W + static_cast<size_t>(16 * p + (l >> 2)) * ld + ks * 16 + 2 * (l & 3);
        return make_uint4(rtc_pred::ld32g(b), rtc_pred::ld32g(b + 8), rtc_pred::ld32g(b + 8 * ld),
                          rtc_pred::ld32g(b + 8 * ld + 8));
    };
    for (int i = tid; i < kSteps1 * 128; i += blockDim.x) reinterpret_cast<uint4*>(sm + SW1)[i] = frag(w.w1_bf16, KP, i);
    for (int i = tid; i < kSteps2 * 128; i += blockDim.x) reinterpret_cast<uint4*>(sm + SW2)[i] = frag(w.w2_bf16, NH, i);
    for (int i = tid; i < NH; i += blockDim.x) {
        reinterpret_cast<float*>(sm + SB1)[i] = w.master[OFF_B1 + i];
        reinterpret_cast<float*>(sm + SB2)[i] = w.master[OFF_B2 + i];
    }
    for (int i = tid; i < NO * NH + NO; i += blockDim.x) reinterpret_cast<float*>(sm + SW3)[i] = w.master[OFF_W3 + i];
    __syncthreads();

    const float inv_sigma = 1.f / sigma;
    const size_t row = 2 * static_cast<size_t>(nv);
    const long long units = static_cast<long long>(tiles) * nk;
    const long long nw = static_cast<long long>(gridDim.x) * (blockDim.x >> 5);
    const long long me = static_cast<long long>(warp) * gridDim.x + blockIdx.x;
    long long u = units * me / nw;
    const long long u1 = units * (me + 1) / nw;

    unsigned char* ring = sm + SRING + warp * 4 * kSlot;
    unsigned char* mine = ring + lane * (kPitch * 4);      // the lane's sample in slot 0
    const uint32_t fragbase = rtc_mvm::smem_addr(ring) + (g * kPitch + t) * 4;
    const uint4* w1s = reinterpret_cast<const uint4*>(sm + SW1) + lane;
    const uint4* w2s = reinterpret_cast<const uint4*>(sm + SW2) + lane;
    const float2* b1s = reinterpret_cast<const float2*>(sm + SB1) + t;
    const float2* b2s = reinterpret_cast<const float2*>(sm + SB2) + t;
    const float2* w3s = reinterpret_cast<const float2*>(sm + SW3) + t;
    const float* b3s = reinterpret_cast<const float*>(sm + SW3) + NO * NH;

    while (u < u1) {
        const int tile = static_cast<int>(u / nk);
        const int kb = k0 + static_cast<int>(u - static_cast<long long>(tile) * nk);
        const int ke = static_cast<int>(min(static_cast<long long>(k0 + nk), kb + (u1 - u)));
        u += ke - kb;
        unsigned off[25];
        const int i0 = tile * kTile;
        {
            const int i = i0 + lane;
#pragma unroll
            for (int nb = 0; nb < 25; ++nb) {
                const int j = i < nv ? __ldg(nbr + static_cast<size_t>(i) * 25 + nb) : -1;
                off[nb] = j >= 0 ? 4u * static_cast<unsigned>(j) : ~0u;
            }
        }
        float v[25];
        for (int k = kb - 3; k <= kb; ++k) {               // fill the ring
            unsigned char* dst = mine + (k & 3) * kSlot;
            load_axis(S + k * row, off, v);
            const uint32_t x24 = store_x(dst, v, inv_sigma);
            load_axis(S + k * row + nv, off, v);
            store_y(dst, v, inv_sigma, x24);
        }
        __syncwarp();
        for (int k = kb; k < ke; ++k) {
            // layer 1: word f / 2 of a sample's features lies in the slot of its lag
            float acc[2][8][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                    for (int h = 0; h < 4; ++h) acc[mt][nt][h] = 0.f;
            uint32_t sl[4];
#pragma unroll
            for (int lag = 0; lag < 4; ++lag) sl[lag] = fragbase + ((k - lag) & 3) * kSlot;
            auto word = [&](int wf0) {                     // address of word wf0 + t
                const int l0 = wf0 / kLagWords, l1 = (wf0 + 3) / kLagWords;
                uint32_t a = sl[l0] + 4 * (wf0 - kLagWords * l0);
                if (l1 != l0 && t >= kLagWords * l1 - wf0) a = sl[l1] + 4 * (wf0 - kLagWords * l1);
                return a;
            };
#pragma unroll
            for (int ks = 0; ks < kSteps1; ++ks) {
                const bool hi = ks * 16 + 8 < rtc_pred::NF;   // the last step's upper half is padding
                const uint32_t pa = word(ks * 8), pb = hi ? word(ks * 8 + 4) : 0u;
                uint32_t a[2][4];
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    a[mt][0] = rtc_mvm::lds32(pa + mt * 16 * kPitch * 4);
                    a[mt][1] = rtc_mvm::lds32(pa + (mt * 16 + 8) * kPitch * 4);
                    a[mt][2] = hi ? rtc_mvm::lds32(pb + mt * 16 * kPitch * 4) : 0u;
                    a[mt][3] = hi ? rtc_mvm::lds32(pb + (mt * 16 + 8) * kPitch * 4) : 0u;
                }
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const uint4 b = w1s[(ks * 4 + p) * 32];
#pragma unroll
                    for (int mt = 0; mt < 2; ++mt) {
                        mma16816(acc[mt][2 * p], a[mt], b.x, b.y);
                        mma16816(acc[mt][2 * p + 1], a[mt], b.z, b.w);
                    }
                }
            }
            __syncwarp();                                  // every lane has read the oldest slot

            // h1 = GELU(z1) as layer 2's A fragments; the next frame's slopes are in
            // flight meanwhile (at the last frame a valid row is read again and stored
            // where nothing is read any more)
            const float* next = S + (k + 1 < ke ? k + 1 : k) * row;
            unsigned char* dst = mine + ((k + 1) & 3) * kSlot;
            uint32_t h1[2][kSteps2][4], x24 = 0;
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                load_axis(next + (mt ? nv : 0), off, v);
#pragma unroll
                for (int nt = 0; nt < 8; ++nt) {
                    const float2 b = b1s[nt * 4];
                    const float2 lo = rtc_pred::gelu2(acc[mt][nt][0] + b.x, acc[mt][nt][1] + b.y);
                    const float2 hi = rtc_pred::gelu2(acc[mt][nt][2] + b.x, acc[mt][nt][3] + b.y);
                    h1[mt][nt >> 1][(nt & 1) * 2] = pack_bf16(lo.x, lo.y);
                    h1[mt][nt >> 1][(nt & 1) * 2 + 1] = pack_bf16(hi.x, hi.y);
                }
                if (mt == 0) x24 = store_x(dst, v, inv_sigma);
                else store_y(dst, v, inv_sigma, x24);
            }

            // layer 2 and the output layer, 16 rows at a time.  Each lane sums its 16 columns
            // in column order, the two row halves packed, then the quad's four sums
            // pairwise (the order of rtc_pred::predict)
            float y[2][2][NO];                             // [mt][row half][output]
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                float acc2[8][4];
#pragma unroll
                for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                    for (int h = 0; h < 4; ++h) acc2[nt][h] = 0.f;
#pragma unroll
                for (int ks = 0; ks < kSteps2; ++ks)
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const uint4 b = w2s[(ks * 4 + p) * 32];
                        mma16816(acc2[2 * p], h1[mt][ks], b.x, b.y);
                        mma16816(acc2[2 * p + 1], h1[mt][ks], b.z, b.w);
                    }
                rtc_pred::f32x2 y0 = rtc_pred::pack2(0.f, 0.f), y1 = y0;
#pragma unroll
                for (int nt = 0; nt < 8; ++nt) {
                    const float2 b = b2s[nt * 4], c0 = w3s[nt * 4], c1 = w3s[NH / 2 + nt * 4];
                    const float2 hx = rtc_pred::gelu2(acc2[nt][0] + b.x, acc2[nt][2] + b.x);
                    const float2 hy = rtc_pred::gelu2(acc2[nt][1] + b.y, acc2[nt][3] + b.y);
                    const rtc_pred::f32x2 px = rtc_pred::pack2(hx.x, hx.y), py = rtc_pred::pack2(hy.x, hy.y);
                    y0 = rtc_pred::fma2(py, rtc_pred::pack2(c0.y, c0.y), rtc_pred::fma2(px, rtc_pred::pack2(c0.x, c0.x), y0));
                    y1 = rtc_pred::fma2(py, rtc_pred::pack2(c1.y, c1.y), rtc_pred::fma2(px, rtc_pred::pack2(c1.x, c1.x), y1));
                }
                const float2 u0 = rtc_pred::unpack2(y0), u1_ = rtc_pred::unpack2(y1);
                y[mt][0][0] = u0.x;
                y[mt][1][0] = u0.y;
                y[mt][0][1] = u1_.x;
                y[mt][1][1] = u1_.y;
            }
            // lane t of the quad keeps row (t >> 1) * 16 + (t & 1) * 8 + g
            float yo[NO];
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                float z[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float s = y[q >> 1][q & 1][o];
                    s += __shfl_xor_sync(0xffffffffu, s, 1);
                    s += __shfl_xor_sync(0xffffffffu, s, 2);
                    z[q] = s;
                }
                yo[o] = (t & 2 ? (t & 1 ? z[3] : z[2]) : (t & 1 ? z[1] : z[0])) + b3s[o];
            }
            const int i = i0 + (t >> 1) * 16 + (t & 1) * 8 + g;
            if (i < nv)
#pragma unroll
                for (int o = 0; o < NO; ++o) {
                    const size_t idx = static_cast<size_t>(o) * nv + i;
                    out[(k + 1) * row + idx] = __fmaf_rn(sigma, yo[o], __ldg(S + k * row + idx));
                }
            __syncwarp();                                  // the new slot is complete
        }
        __syncwarp();                                      // the ring may be refilled
    }
}

}  // namespace

cudaError_t mlp_predict_configure() {
    return cudaFuncSetAttribute(mlp_predict_seq_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                smem_bytes(kMaxWarps));
}

cudaError_t mlp_launch_predict(const MlpDev& w, const float* S, float* out, int k0, int nk, int nv, const int* nbr,
                               float sigma, int sms, cudaStream_t st) {
    if (nv == 0 || nk <= 0) return cudaSuccess;
    const int tiles = (nv + kTile - 1) / kTile;
    // as many warps as there are units, spread over the SMs; at least 4 a block, which
    // share the weight loads
    const long long units = static_cast<long long>(tiles) * nk;
    const int blocks = static_cast<int>(std::min<long long>(units, sms));
    const int warps = static_cast<int>(std::min<long long>(kMaxWarps, std::max<long long>(4, (units + blocks - 1) / blocks)));
    mlp_predict_seq_kernel<<<blocks, warps * 32, smem_bytes(warps), st>>>(w, S, out, k0, nk, nv, nbr, sigma, tiles);
    return cudaGetLastError();
}
