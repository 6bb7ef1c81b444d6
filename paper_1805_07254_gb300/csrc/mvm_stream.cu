// The sum of the partial DM vectors, and the stand-alone reconstruction (d = M s and the
// leaky integrator, Fig. 3 (c)-(d)) on a full slope vector.
//
// A per-frame call is two kernels: one writes a partial DM vector per matrix slice
// (frame_kernel.cu, or mvm_stream_kernel here for rtc_reconstruct_async), the other
// sums them (mvm_reduce_kernel).  The end of the first kernel is the barrier between
// them, so no block ever waits for another one: nothing has to be co-resident, and the
// launches need not be cooperative ones, which start only on an idle device.  Both are
// launched with programmatic dependent launch and let their successor start at once:
//   - the sum's blocks are small enough to sit on the SMs beside the streaming blocks
//     and wait there, in hardware, for the partials;
//   - the next frame's streaming blocks start as soon as this frame's leave their SM:
//     their set-up and their first matrix tiles (none or one for most frames, the whole
//     ring for some: plan_launch, stream_mvm.cuh) run during the slowest blocks, the sum,
//     and the hand-over, and they wait only before they read pixels.
// Everything a kernel reads before its wait is written by no kernel (matrix, slice
// table, maps, row scales).  frame_kernel.cu has the figures of this and of one
// cooperative kernel with a grid barrier, whose launch waited for an idle device.

#include "launch.cuh"
#include "pred_tile.cuh"
#include "stream_mvm.cuh"

namespace {

using namespace rtc_mvm;

template <int DT, bool CHAIN>
__global__ void __launch_bounds__(kFrameRegThreads, 1) mvm_stream_kernel(Args g) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ Shared sh;
    const int tid = threadIdx.x;
    pdl_launch_dependents();
    if (tid == 0) init_shared(sh);
    __syncthreads();
    const Plan pl = make_plan(g, smem);
    if (tid >= kConsumers) {
        if ((tid & 31) == 0) produce(g, pl, sh);
        return;
    }
    clear_local(g, pl, tid);
    consumer_sync();
    pdl_wait();
    gather_local(g, pl, tid, g.s, true);
    consumer_sync();
    consume<DT, CHAIN>(g, pl, sh, tid, 0);
}

// 32 rows a block, one per lane; the order of reduce_rows (stream_mvm.cuh).  A step that
// a bounded wait cut short (its own mark: record_timeout) leaves the integrator as it
// was, and the last block to have read the mark clears it for the next step.  HOST: the
// last block to finish writes the caller's completion record.
template <bool HOST>
__global__ void __launch_bounds__(kConsumers, 4) mvm_reduce_kernel(SumArgs r, FrameHost fh) {
    __shared__ float red[kConsumerWarps * 32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int row = blockIdx.x * 32 + lane;
    pdl_launch_dependents();
    const bool mine = warp == 0 && row < r.nact;
    const float sc = mine && r.scale ? __ldg(r.scale + row) : 1.f;
    pdl_wait();
    float a_prev = 0.f;
    int cut = RTC_OK;
    if (mine) {
        a_prev = __ldcg(r.a + row);
        cut = *reinterpret_cast<volatile int*>(r.cut);
    }
    // the warp's slices w, w + 14, ...: 11 in flight (152 slices are one round)
    constexpr int kFlight = 11;
    float v = 0.f;
    if (row < r.nact) {
        for (int s0 = warp; s0 < r.S; s0 += kFlight * kConsumerWarps) {
            float p[kFlight];
#pragma unroll
            for (int j = 0; j < kFlight; ++j) {
                const int s = s0 + j * kConsumerWarps;
                p[j] = s < r.S ? __ldcg(r.partial + static_cast<size_t>(s) * r.pitch + row) : 0.f;
            }
#pragma unroll
            for (int j = 0; j < kFlight; ++j)
                if (s0 + j * kConsumerWarps < r.S) v += p[j];
        }
    }
    red[warp * 32 + lane] = v;
    __syncthreads();
    // (here: with it at the kernel's end frames one after another took up to 0.4 us more,
    // and frames from the host, here, 0.2 us)
    auto clear = [&]() {
        if (tid == 0 && cut != RTC_OK && atomicInc(r.cutctr, gridDim.x - 1) == gridDim.x - 1) *r.cut = RTC_OK;
    };
    if (!HOST) clear();
    if (mine && cut == RTC_OK) {
        float t[kConsumerWarps];
#pragma unroll
        for (int w = 0; w < kConsumerWarps; ++w) t[w] = red[w * 32 + lane];
#pragma unroll
        for (int width = 1; width < kConsumerWarps; width <<= 1)
#pragma unroll
            for (int i = 0; i + width < kConsumerWarps; i += 2 * width) t[i] += t[i + width];
        const float d = r.scale ? t[0] * sc : t[0];
        const float an = fmaf(r.leak, a_prev, r.gain * d);
        r.a[row] = an;
        if (r.dm_out) r.dm_out[row] = an;
    }
    if (HOST) clear();
    if (HOST) {
        __syncthreads();
        if (tid == 0) finish_host(fh, r.status);
    }
}

// With no slopes, d = 0: only the leak acts.
__global__ void decay_kernel(int nact, float* __restrict__ a, float* __restrict__ dm_out,
                             float leak) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nact) {
        const float an = leak * a[i];
        a[i] = an;
        if (dm_out) dm_out[i] = an;
    }
}

template <int DT>
cudaError_t launch_stream(rtc_handle* h, const float* d_s, float* d_dm_out, cudaStream_t st) {
    const Launch& L = frame_plan(h, rtc_pred::kSmemBytes, false);
    if (!L.ok) return cudaErrorInvalidValue;
    const Args g = make_args(h, d_s, L);
    const auto k = L.chain ? mvm_stream_kernel<DT, CanChain<DT>::v> : mvm_stream_kernel<DT, false>;
    const cudaError_t e = launch_pdl(k, dim3(L.G), dim3(kThreads), L.smem, st, g);
    return e == cudaSuccess ? launch_sum(h, d_dm_out, st) : e;
}

template <int DT>
cudaError_t configure_one() {
    const int bytes = static_cast<int>(kDynSmemBudget);
    const cudaError_t e =
        cudaFuncSetAttribute(mvm_stream_kernel<DT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess || !CanChain<DT>::v) return e;
    return cudaFuncSetAttribute(mvm_stream_kernel<DT, CanChain<DT>::v>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                bytes);
}

}  // namespace

rtc_mvm::SumArgs sum_args(const rtc_handle* h, float* d_dm_out) {
    const bool scaled = h->store == RTC_FP8_E4M3 || h->store == RTC_INT8;
    return SumArgs{h->d_partial, scaled ? h->d_scale : nullptr, h->d_a,       d_dm_out,
                   h->d_status,  h->d_status + 1,               h->d_lastctr, h->sl_S,
                   h->cfg.nact,  partial_pitch(h->cfg.nact),    h->gain,      h->leak};
}

cudaError_t launch_sum(rtc_handle* h, float* d_dm_out, cudaStream_t st, FrameHost* fh) {
    const SumArgs r = sum_args(h, d_dm_out);
    const dim3 grid((h->cfg.nact + 31) / 32), block(kConsumers);
    if (!fh) {
        // In a server slot with a matrix that comes from the HBM every frame, the sum starts
        // when the stream is done: the SMs have room for one job's waiting blocks beside
        // the streaming ones, and those of other jobs would queue up behind them for the
        // whole of its long stream (four ELT FP32 jobs 30.2 us a frame, so 28.4).  Other
        // slots gain from the early start (eight 41x41 FP16 jobs 12.9 against 13.7).
        const bool overlap = !h->in_slot || h->m_bytes <= kL2KeepBytes;
        return launch_pdl_if(overlap, mvm_reduce_kernel<false>, grid, block, 0, st, r, FrameHost{});
    }
    fh->target = h->pf_arrivals + grid.x;
    const cudaError_t e = launch_pdl(mvm_reduce_kernel<true>, grid, block, 0, st, r, *fh);
    if (e == cudaSuccess) h->pf_arrivals = fh->target;
    return e;
}

cudaError_t mvm_stream_configure() {
    cudaError_t e = configure_one<RTC_F32>();
    if (e == cudaSuccess) e = configure_one<RTC_BF16>();
    if (e == cudaSuccess) e = configure_one<RTC_F16>();
    if (e == cudaSuccess) e = configure_one<RTC_FP8_E4M3>();
    if (e == cudaSuccess) e = configure_one<RTC_INT8>();
    return e;
}

cudaError_t launch_decay(const rtc_handle* h, float* d_dm_out, cudaStream_t st) {
    decay_kernel<<<(h->cfg.nact + 255) / 256, 256, 0, st>>>(h->cfg.nact, h->d_a, d_dm_out, h->leak);
    return cudaGetLastError();
}

cudaError_t launch_mvm_integrate(rtc_handle* h, const float* d_s, float* d_dm_out, cudaStream_t st) {
    if (h->kpad == 0) return launch_decay(h, d_dm_out, st);
    switch (h->store) {
        case RTC_F32: return launch_stream<RTC_F32>(h, d_s, d_dm_out, st);
        case RTC_BF16: return launch_stream<RTC_BF16>(h, d_s, d_dm_out, st);
        case RTC_F16: return launch_stream<RTC_F16>(h, d_s, d_dm_out, st);
        case RTC_FP8_E4M3: return launch_stream<RTC_FP8_E4M3>(h, d_s, d_dm_out, st);
        case RTC_INT8: return launch_stream<RTC_INT8>(h, d_s, d_dm_out, st);
        default: return cudaErrorInvalidValue;
    }
}
