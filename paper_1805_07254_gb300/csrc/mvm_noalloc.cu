// Reconstruction + integrator for callers that cannot allocate device memory.
//
// Some hosts of this code must never call cudaMalloc: a hard-real-time control
// thread cannot risk the implicit device synchronisation and unbounded latency
// of the allocator inside its loop, and a plugin embedded in a larger RTC
// framework may be handed all of its device buffers by that framework and be
// forbidden to allocate its own.  rtc_mvm_integrate_noalloc serves them: it runs
// d = M s and a <- leak * a + gain * d on the caller's row-major [nact][kpad] matrix.
//
// What bounds it: the matrix bytes (an FP32 one of 5169 x 9424 is 195 MB, 28.7 us at the
// measured copy rate).  So each SM gets one block and an equal run of consecutive
// rows -- a contiguous part of the matrix, streamed by bulk copies through a ring in
// shared memory, with no block waiting for another and no scratch in device memory.
// The slopes are the same for every row: a thread's share of them (32 floats) stays in
// its registers, so a row costs one shared-memory read and the FMAs.  `wpr` warps share
// a row, the fewest whose registers hold all slopes (1, 2, 7 or the block's 14), so short
// rows go several at a time; rows beyond 14,336 elements are done in panels of that
// width.  A row's sum is short chains and a pairwise tree per thread, a butterfly over the
// warp and a tree over the row's warps: it depends on neither the SM count nor `ksplit`
// (the number of column splits asked for, which this kernel does not need).
//
// Measured, 5169 x 9416 FP32, call after call: 31.0 us, 6.3 TB/s (42.3 us with 1293 blocks
// of 4 rows and 256 threads, 2.1 waves of them, the splits' partial sums in a static
// device array and a memset of their counters per call).

#include <mutex>

#include "launch.cuh"
#include "stream_mvm.cuh"

namespace {

using namespace rtc_mvm;

constexpr int kSlopesPerThread = 32;
constexpr int kTileTarget = 48 * 1024;
constexpr int kMaxRows = 256;                  // rows of a block, at most

struct NoallocArgs {
    const unsigned char* M;   // [nact][kpad]
    const float* s;           // [kpad]
    const float* scale;       // [nact] or null
    float* a;                 // [nact]
    float* dm_out;            // [nact] or null
    int nact, kpad;
    int wpr;                  // warps a row: 1, 2, 7 or 14
    int rt;                   // rows a tile
    int stage_s;              // the slopes go through shared memory (wpr 1 and 2)
    int nst, stage_bytes;
    int l2_policy;
    float gain, leak;
};

// One 16-byte chunk of a row with its slopes, as two short chains.
template <int DT>
__device__ __forceinline__ float chunk_dot(const uint4& m, const float* sv) {
    constexpr int EPW = 4 / Esize<DT>::v;
    return word_dot<DT>(word_dot<DT>(0.f, m.x, sv), m.y, sv + EPW) +
           word_dot<DT>(word_dot<DT>(0.f, m.z, sv + 2 * EPW), m.w, sv + 3 * EPW);
}

template <int DT>
__global__ void __launch_bounds__(kThreads, 1) mvm_noalloc_kernel(NoallocArgs g) {
    constexpr int ES = Esize<DT>::v, E = 16 / ES, C = kSlopesPerThread / E;   // elements a 16-byte chunk, chunks
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ Shared sh;
    const int tid = threadIdx.x;
    const int r0 = static_cast<int>(static_cast<long long>(g.nact) * blockIdx.x / gridDim.x);
    const int r1 = static_cast<int>(static_cast<long long>(g.nact) * (blockIdx.x + 1) / gridDim.x);
    const int tpr = g.wpr * 32;                              // threads a row
    const int chunks = g.kpad / E, pch = tpr * C;            // chunks of a row, of a panel
    const size_t pitch = static_cast<size_t>(g.kpad) * ES;
    const uint32_t ring = smem_addr(smem);
    float* red = reinterpret_cast<float*>(smem + static_cast<size_t>(g.nst) * g.stage_bytes);
    pdl_launch_dependents();
    if (tid == 0) init_shared(sh);
    __syncthreads();
    pdl_wait();                                              // the caller's buffers
    if (tid >= kConsumers) {
        if ((tid & 31) != 0) return;
        const unsigned long long policy = matrix_policy(g.l2_policy);
        int t = 0;
        bool ok = true;
        for (int c0 = 0; c0 < chunks && ok; c0 += pch) {
            const uint32_t rowb = min(pch, chunks - c0) * 16u;
            for (int row = r0; row < r1; row += g.rt, ++t) {
                const int st = t % g.nst, use = t / g.nst, n = min(g.rt, r1 - row);
                if (use > 0 && !wait_phase(smem_addr(&sh.empty_bar[st]), (use - 1) & 1, &sh.abort_flag)) {
                    ok = false;
                    break;
                }
                // whole rows are contiguous; with panels a tile is one row's part (rt = 1)
                const uint32_t fb = smem_addr(&sh.full_bar[st]), bytes = n * rowb;
                const unsigned char* src = g.M + row * pitch + static_cast<size_t>(c0) * 16;
                mbar_expect_tx(fb, bytes);
                for (uint32_t o = 0; o < bytes; o += kCopyBytes)
                    bulk_g2s(ring + st * g.stage_bytes + o, src + o, min(kCopyBytes, bytes - o), fb, policy);
            }
        }
        if (!ok) sh.abort_flag = 1;
        for (int k = max(0, t - g.nst); k < t; ++k)          // no copy in flight at exit
            wait_phase(smem_addr(&sh.full_bar[k % g.nst]), (k / g.nst) & 1, nullptr);
        return;
    }
    // Where many warps of a block want the same slopes, they come once, and into an order in
    // which a thread's share (E floats at a stride of E) is read without bank conflicts.
    // (With every warp of every SM reading the same few lines of L2 the reads queued up
    // there: 300 x 300 FP8 took 9.8 us a call, 5169 x 160 INT8 8.6; now 4.1 and 4.2, which
    // is the host's time.)
    const float4* s4 = reinterpret_cast<const float4*>(g.s);
    float4* staged = reinterpret_cast<float4*>(red + ((r1 - r0) * g.wpr + 3) / 4 * 4);
    auto swizzled = [](int i) { return i ^ ((i >> 3) & 3); };
    if (g.stage_s) {
        for (int i = tid; i < g.kpad / 4; i += kConsumers) staged[swizzled(i)] = __ldcg(s4 + i);
        consumer_sync();
    }
    const int rg = tid / tpr, ts = tid - rg * tpr, lane = tid & 31, nrg = kConsumerWarps / g.wpr;
    int st = 0, phase = 0;
    for (int c0 = 0; c0 < chunks; c0 += pch) {
        const int nch = min(pch, chunks - c0);
        float sv[C][E];
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const int c = ts + j * tpr;
#pragma unroll
            for (int e = 0; e < E; e += 4) {
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                const int i = (c0 + c) * (E / 4) + e / 4;
                if (c < nch) v = g.stage_s ? staged[swizzled(i)] : __ldcg(s4 + i);
                sv[j][e] = v.x;
                sv[j][e + 1] = v.y;
                sv[j][e + 2] = v.z;
                sv[j][e + 3] = v.w;
            }
        }
        for (int row = r0; row < r1; row += g.rt) {
            const bool ok = __all_sync(0xffffffffu, wait_phase(smem_addr(&sh.full_bar[st]), phase, &sh.abort_flag));
            if (ok) {
                const int n = min(g.rt, r1 - row);
                for (int r = rg; r < n; r += nrg) {
                    const uint32_t at = ring + st * g.stage_bytes + (r * nch + ts) * 16;
                    uint4 m[C];
#pragma unroll
                    for (int j = 0; j < C; ++j) {
                        m[j] = make_uint4(0u, 0u, 0u, 0u);
                        if (ts + j * tpr < nch) m[j] = lds128(at + j * tpr * 16);
                    }
                    float d[C];
#pragma unroll
                    for (int j = 0; j < C; ++j) d[j] = ts + j * tpr < nch ? chunk_dot<DT>(m[j], sv[j]) : 0.f;
#pragma unroll
                    for (int width = 1; width < C; width <<= 1)
#pragma unroll
                        for (int j = 0; j < C; j += 2 * width) d[j] += d[j + width];
                    float acc = d[0];
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
                    if (lane == 0) {
                        float* p = red + (row - r0 + r) * g.wpr + (ts >> 5);
                        *p = c0 ? *p + acc : acc;
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_addr(&sh.empty_bar[st]));
            } else if (lane == 0) {
                sh.abort_flag = 1;
            }
            if (++st == g.nst) {
                st = 0;
                phase ^= 1;
            }
        }
    }
    consumer_sync();
    for (int i = tid; i < r1 - r0; i += kConsumers) {
        const int row = r0 + i;
        float t[kConsumerWarps];
#pragma unroll
        for (int w = 0; w < kConsumerWarps; ++w) t[w] = chunks > 0 && w < g.wpr ? red[i * g.wpr + w] : 0.f;
#pragma unroll
        for (int width = 1; width < kConsumerWarps; width <<= 1)
#pragma unroll
            for (int w = 0; w + width < kConsumerWarps; w += 2 * width) t[w] += t[w + width];
        const float d = RowScaled<DT>::v ? t[0] * g.scale[row] : t[0];
        float an = fmaf(g.leak, g.a[row], g.gain * d);
        // a copy that never landed: the command is not a number, the state stays as it
        // was, so that the next call starts from it
        if (sh.abort_flag) an = __uint_as_float(0x7fc00000u);
        else g.a[row] = an;
        if (g.dm_out) g.dm_out[row] = an;
    }
}

constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
int g_sms[kMaxDevices] = {};

template <int DT>
cudaError_t configure() {
    return cudaFuncSetAttribute(mvm_noalloc_kernel<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(kDynSmemBudget));
}

template <int DT>
cudaError_t launch_t(NoallocArgs g, int sms, cudaStream_t st) {
    constexpr int es = Esize<DT>::v;
    // the fewest warps a row whose threads hold its slopes
    const int per_warp = 32 * kSlopesPerThread;
    g.wpr = g.kpad <= per_warp ? 1 : g.kpad <= 2 * per_warp ? 2 : g.kpad <= 7 * per_warp ? 7 : kConsumerWarps;
    const int panel = g.wpr * per_warp, nrg = kConsumerWarps / g.wpr;
    const bool panels = g.kpad > panel;
    const int rowb = std::max(16, std::min(g.kpad, panel) * es);
    const int blocks = std::max(std::min(g.nact, sms), (g.nact + kMaxRows - 1) / kMaxRows);
    const int rows = (g.nact + blocks - 1) / blocks;
    // tiles of about 48 KB, whole rounds of the row groups, and no more shared memory than
    // the block's rows fill
    g.rt = panels ? 1 : std::min(rows, nrg * std::max(1, kTileTarget / (nrg * rowb)));
    g.stage_bytes = (g.rt * rowb + 127) / 128 * 128;
    g.stage_s = g.wpr <= 2;
    const size_t red = (static_cast<size_t>(rows) * g.wpr + 3) / 4 * 16;
    const size_t extra = red + (g.stage_s ? (g.kpad / 4 + 7) / 8 * 8 * sizeof(float4) : 0);
    const int tiles = (rows + g.rt - 1) / g.rt * std::max(1, (g.kpad + panel - 1) / panel);
    g.nst = std::min(std::min(8, tiles), static_cast<int>((kDynSmemBudget - extra) / g.stage_bytes));
    const size_t smem = static_cast<size_t>(g.nst) * g.stage_bytes + extra;
    g.l2_policy = static_cast<long long>(g.nact) * g.kpad * es <= kL2KeepBytes ? kL2Normal : kL2Stream;
    return launch_pdl(mvm_noalloc_kernel<DT>, dim3(blocks), dim3(kThreads), smem, st, g);
}

int noalloc_fail(int code, const char* msg) {
    rtc_set_global_error(msg);
    return code;
}

}  // namespace

extern "C" int rtc_mvm_integrate_noalloc(const void* d_M, int32_t store, const float* d_row_scales,
                                         int32_t nact, int32_t kpad, const float* d_s, float* d_a,
                                         float* d_dm_out, float gain, float leak, int32_t ksplit,
                                         void* stream) {
    if (nact <= 0 || nact > RTC_NOALLOC_MAX_NACT)
        return noalloc_fail(RTC_EINVAL, "nact must be in 1..RTC_NOALLOC_MAX_NACT (8192)");
    if (ksplit < 1 || ksplit > RTC_NOALLOC_MAX_KSPLIT)
        return noalloc_fail(RTC_EINVAL, "ksplit must be in 1..RTC_NOALLOC_MAX_KSPLIT (16)");
    if (kpad < 0 || kpad % 16 != 0) return noalloc_fail(RTC_EINVAL, "kpad must be a multiple of 16");
    if (store != RTC_F32 && store != RTC_BF16 && store != RTC_F16 && store != RTC_FP8_E4M3 &&
        store != RTC_INT8)
        return noalloc_fail(RTC_EINVAL, "unknown store type");
    if (!d_s || !d_a || (kpad > 0 && !d_M)) return noalloc_fail(RTC_EINVAL, "NULL buffer");
    if ((store == RTC_FP8_E4M3 || store == RTC_INT8) && !d_row_scales)
        return noalloc_fail(RTC_EINVAL, "FP8 and INT8 need row scales");
    if ((reinterpret_cast<uintptr_t>(d_M) | reinterpret_cast<uintptr_t>(d_s)) & 15)
        return noalloc_fail(RTC_EINVAL, "d_M and d_s must be 16-byte aligned");

    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
        return noalloc_fail(RTC_EDEVICE, "no usable current CUDA device");
    int sms;
    {
        // the kernels' shared-memory limit and the SM count, once per device
        std::lock_guard<std::mutex> lock(g_setup_mutex);
        if (!g_sms[dev]) {
            int n = 0;
            cudaError_t e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess) e = configure<RTC_F32>();
            if (e == cudaSuccess) e = configure<RTC_BF16>();
            if (e == cudaSuccess) e = configure<RTC_F16>();
            if (e == cudaSuccess) e = configure<RTC_FP8_E4M3>();
            if (e == cudaSuccess) e = configure<RTC_INT8>();
            if (e != cudaSuccess || n < 1) return noalloc_fail(RTC_EDEVICE, cudaGetErrorString(e));
            g_sms[dev] = n;
        }
        sms = g_sms[dev];
    }
    const NoallocArgs g{static_cast<const unsigned char*>(d_M), d_s, d_row_scales, d_a, d_dm_out, nact, kpad, 0, 0, 0,
                        0, 0, 0, gain, leak};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaErrorInvalidValue;
    switch (store) {
        case RTC_F32: e = launch_t<RTC_F32>(g, sms, st); break;
        case RTC_BF16: e = launch_t<RTC_BF16>(g, sms, st); break;
        case RTC_F16: e = launch_t<RTC_F16>(g, sms, st); break;
        case RTC_FP8_E4M3: e = launch_t<RTC_FP8_E4M3>(g, sms, st); break;
        case RTC_INT8: e = launch_t<RTC_INT8>(g, sms, st); break;
    }
    if (e != cudaSuccess) return noalloc_fail(RTC_EDEVICE, cudaGetErrorString(e));
    return RTC_OK;
}
