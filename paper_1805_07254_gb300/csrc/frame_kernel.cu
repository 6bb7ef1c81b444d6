// The per-frame path of Sec. 2.1 / Fig. 3: pixels -> slopes -> partial DM vectors in one
// kernel, their sum and the integrator in a second (mvm_reduce_kernel, mvm_stream.cu,
// which also says how the two overlap with each other and with the next frame's).
//
// Each block owns a run of matrix slices (stream_mvm.cuh) and the subapertures
// whose slopes those slices multiply.  While its producer warp streams the slices'
// matrix tiles into shared memory (the matrix does not depend on the frame), the
// consumer warps compute the block's slopes (pixel.cuh) into shared memory and
// multiply them straight away: no block waits for another, as in the paper's
// per-thread column blocks (Sec. 2.3).  Each block writes one partial DM vector per
// slice.  The producer starts at once, before the previous kernel of the stream has
// finished, and so do the subaperture positions and the calibration data; the block
// waits for its predecessor before it reads pixels.
//
// With the learned slope predictor on, the measured slopes of all blocks have to be
// known before any can predict, so the pixel stage is a kernel of its own: it writes
// the slopes into the history ring (calib_cog.cu; frame_slopes_kernel for a frame in
// host memory), and frame_pred_kernel predicts the next slopes of its own subapertures
// from their neighbourhoods (pred_tile.cuh, in the shared scratch before the slopes),
// writing them straight into its local slope vector, and multiplies those.
//
// For rtc_process_frame with pinned host buffers (HOST) the frame is read in place
// from mapped host memory and the sum kernel writes the DM commands there and the
// caller's completion record, so the host needs no copies and no stream
// synchronisation.
//
// Measured, frame after frame on one stream (one cooperative kernel with a grid barrier
// -> this): ELT FP32 28.9 -> 25.4 us, INT8 20.9 -> 17.0, BF16 with prediction 28.4 ->
// 27.1, six ELT sensors FP8 59.4 -> 54.6, 41x41 FP16 12.3 -> 7.6 and 8x8 FP32 10.3 -> 6.2
// (GPU time; the two launches' host time, 4 us in the library, bounds the last two).  Of
// an FP32 frame the blocks stream 17 us (6.5 TB/s); slopes are known 2.9 us after the
// last frame's sum, the hand-over to the sum takes 0.9 us and the sum 1.4.

#include "launch.cuh"
#include "mlp.h"
#include "pixel.cuh"
#include "pred_tile.cuh"
#include "stream_mvm.cuh"

namespace {

using namespace rtc_mvm;

// The block's subapertures, one half-warp each (the ~26 of an ELT block are a single
// round), into the slope vectors and, if LOCAL, the block's local one.  The first round's
// pixel lines are brought into L2 before the wait (a frame that a matrix stream has
// evicted costs an HBM round trip otherwise: ELT INT8 13.5 against 13.8 us).  HOST: the
// block's pixel rows first go from mapped host memory into device staging, in 16-byte
// units over the host link, and are read through L2.  pos0: grid position of the
// thread's first subaperture.
template <int NPX, bool HOST, bool LOCAL>
__device__ __forceinline__ void pixel_stage(const rtc_pixel::PixelArgs& px, const Args& g, const Plan& pl,
                                            const FrameHost& fh, int slot, int2 pos0, int tid) {
    if (!HOST) rtc_pixel::prefetch_rows_l2(px, pl.g0 + slot, pl.g0 + slot < pl.g1, pos0, tid);
    if (HOST) {
        pdl_wait();
        rtc_pixel::ingest_block<kConsumers>(px.frame, fh.stage, fh.units, __ldg(fh.blk + blockIdx.x), fh.unit,
                                            tid);
        consumer_sync();
    }
    const uint16_t* frame = HOST ? fh.stage : px.frame;
    for (int base = pl.g0; base < pl.g1; base += 2 * kConsumerWarps) {
        const int gi = base + slot;
        const bool valid = gi < pl.g1;
        const int2 pos = base == pl.g0 ? pos0 : rtc_pixel::subap_pos(px, gi, valid);
        const float2 sxy = rtc_pixel::subap_slopes_at<NPX, rtc_pixel::kPixelL2, 16>(
            px, frame, px.s, gi, valid, tid & 31, pos, rtc_pixel::NoHook(), pdl_wait);
        if (LOCAL && valid && (tid & 15) == 0) {
            int ix, iy;
            local_index(g, pl, gi, ix, iy);
            pl.loc[ix] = sxy.x;
            pl.loc[iy] = sxy.y;
        }
    }
}

template <int DT, int NPX, bool HOST>
__global__ void __launch_bounds__(kFrameRegThreads, 1)
frame_kernel(rtc_pixel::PixelArgs px, Args g, FrameHost fh) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ Shared sh;
    const int tid = threadIdx.x;
    pdl_launch_dependents();
    const Plan pl = make_plan(g, smem);
    // the grid position of a consumer's first subaperture, loaded before the
    // block's set-up so that its latency overlaps it
    const int slot = 2 * (tid >> 5) + ((tid >> 4) & 1);
    const int2 pos0 = rtc_pixel::subap_pos(px, pl.g0 + slot, tid < kConsumers && pl.g0 + slot < pl.g1);
    if (tid == 0) init_shared(sh);
    __syncthreads();
    if (tid >= kConsumers) {
        if ((tid & 31) == 0) produce(g, pl, sh);
        return;
    }
    clear_local(g, pl, tid);
    consumer_sync();
    pixel_stage<NPX, HOST, true>(px, g, pl, fh, slot, pos0, tid);
    pdl_wait();                         // before the partials of the last frame are overwritten
    consumer_sync();
    consume<DT>(g, pl, sh, tid, 0);
}

// The pixel stage alone, for a frame in host memory and the predictor.
template <int NPX>
__global__ void __launch_bounds__(kThreads, 1) frame_slopes_kernel(rtc_pixel::PixelArgs px, Args g, FrameHost fh) {
    const int tid = threadIdx.x;
    pdl_launch_dependents();
    if (tid >= kConsumers) return;
    const Plan pl = make_plan(g, nullptr);
    const int slot = 2 * (tid >> 5) + ((tid >> 4) & 1);
    const int2 pos0 = rtc_pixel::subap_pos(px, pl.g0 + slot, pl.g0 + slot < pl.g1);
    pixel_stage<NPX, true, false>(px, g, pl, fh, slot, pos0, tid);
}

// Prediction and multiplication: the measured slopes are in ring row `head`, written by
// the kernel before this one.  That kernel lets this one start at once, so that the ring
// fills and the network's weights arrive while the pixel stage waits for the frame; the
// history is read after the wait.
template <int DT>
__global__ void __launch_bounds__(kFrameRegThreads, 1) frame_pred_kernel(Args g, rtc_pred::PredArgs pa, int head) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ Shared sh;
    const int tid = threadIdx.x;
    pdl_launch_dependents();
    const Plan pl = make_plan(g, smem);
    if (tid == 0) init_shared(sh);
    __syncthreads();
    if (tid >= kConsumers) {
        if ((tid & 31) == 0) produce(g, pl, sh);
        return;
    }
    clear_local(g, pl, tid);
    rtc_pred::Regs pr;
    rtc_pred::prefetch<false>(pa, pl.scratch, tid, pl.g0, pl.g1, head, pr);
    consumer_sync();
    pdl_wait();
    const float* s_k = pa.ring + static_cast<size_t>(head) * pa.kpad;
    rtc_pred::predict<false>(
        pa, pl.scratch, tid, pl.g0, pl.g1, head, pr,
        [&](int gi, int axis) { return __ldcg(s_k + axis * pa.nv + gi); },
        [&](int gi, int axis, float v) {
            int ix, iy;
            local_index(g, pl, gi, ix, iy);
            pl.loc[axis ? iy : ix] = v;
        });
    consumer_sync();
    consume<DT>(g, pl, sh, tid, 0);
}

template <int DT, bool HOST>
cudaError_t launch_npx(const rtc_handle* h, const Launch& L, const rtc_pixel::PixelArgs& px, const Args& g,
                       const FrameHost& fh, cudaStream_t st) {
    const dim3 grid(L.G), block(kThreads);
    if (h->cfg.npx == 10) return launch_pdl(frame_kernel<DT, 10, HOST>, grid, block, L.smem, st, px, g, fh);
    return launch_pdl(frame_kernel<DT, 0, HOST>, grid, block, L.smem, st, px, g, fh);
}

template <int DT>
cudaError_t launch_dt(rtc_handle* h, const uint16_t* d_frame, float* d_dm_out, float* d_s_meas,
                      int head, cudaStream_t st, FrameHost* fh, float* d_s2) {
    const bool pred = d_s_meas != nullptr;
    const Launch& L = frame_plan(h, rtc_pred::kSmemBytes, pred);
    if (!L.ok) return cudaErrorInvalidValue;
    const rtc_pixel::PixelArgs px = pixel_args(h, d_frame, pred ? d_s_meas : h->d_s, d_s2);
    const Args g = make_args(h, h->d_s, L);
    if (fh) {
        // the copy units of each block's pixel rows (16 bytes when the frame allows)
        const size_t fbytes = static_cast<size_t>(h->cfg.n_wfs) * h->side * h->side * 2;
        const uintptr_t bases = reinterpret_cast<uintptr_t>(d_frame) | reinterpret_cast<uintptr_t>(h->d_frame);
        fh->unit = (fbytes % 16 == 0 && bases % 16 == 0) ? 16 : (fbytes % 4 == 0 && bases % 4 == 0) ? 4 : 2;
        const int rc = build_ingest(h, L.G, fh->unit, 1);
        if (rc == RTC_ENOMEM) return cudaErrorMemoryAllocation;
        if (rc != RTC_OK) return cudaErrorUnknown;
        fh->units = h->d_units;
        fh->blk = h->d_blk;
        fh->stage = h->d_frame;
    }
    cudaError_t e;
    if (!pred) {
        e = fh ? launch_npx<DT, true>(h, L, px, g, *fh, st) : launch_npx<DT, false>(h, L, px, g, FrameHost{}, st);
    } else {
        if (!fh) e = launch_calib_cog(h, d_frame, d_s_meas, d_s2, true, st);
        else if (h->cfg.npx == 10) e = launch_pdl(frame_slopes_kernel<10>, dim3(L.G), dim3(kThreads), 0, st, px, g, *fh);
        else e = launch_pdl(frame_slopes_kernel<0>, dim3(L.G), dim3(kThreads), 0, st, px, g, *fh);
        if (e == cudaSuccess)
            e = launch_pdl(frame_pred_kernel<DT>, dim3(L.G), dim3(kThreads), L.smem, st, g, pred_args(h), head);
    }
    return e == cudaSuccess ? launch_sum(h, d_dm_out, st, fh) : e;
}

template <typename K>
cudaError_t configure(K kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kDynSmemBudget));
}

template <int DT>
cudaError_t configure_dt() {
    cudaError_t e = configure(frame_kernel<DT, 10, false>);
    if (e == cudaSuccess) e = configure(frame_kernel<DT, 0, false>);
    if (e == cudaSuccess) e = configure(frame_kernel<DT, 10, true>);
    if (e == cudaSuccess) e = configure(frame_kernel<DT, 0, true>);
    if (e == cudaSuccess) e = configure(frame_pred_kernel<DT>);
    return e;
}

}  // namespace

cudaError_t frame_kernel_configure() {
    cudaError_t e = configure_dt<RTC_F32>();
    if (e == cudaSuccess) e = configure_dt<RTC_BF16>();
    if (e == cudaSuccess) e = configure_dt<RTC_F16>();
    if (e == cudaSuccess) e = configure_dt<RTC_FP8_E4M3>();
    if (e == cudaSuccess) e = configure_dt<RTC_INT8>();
    return e;
}

rtc_pred::PredArgs pred_args(const rtc_handle* h) {
    rtc_pred::PredArgs pa{};
    pa.w1 = h->pred->w1_bf16;
    pa.w2 = h->pred->w2_bf16;
    pa.params = h->pred->master;
    pa.nbr = h->d_nbr;
    pa.ring = h->d_ring;
    pa.s_pred = h->d_spred;
    pa.kpad = h->kpad;
    pa.nv = h->n_valid;
    pa.sigma = h->pred_sigma;
    pa.inv_sigma = 1.f / h->pred_sigma;
    return pa;
}

cudaError_t launch_frame(rtc_handle* h, const uint16_t* d_frame, float* d_dm_out, float* d_s_meas,
                         int head, cudaStream_t st, FrameHost* fh, float* d_s2) {
    if (h->kpad == 0) return launch_decay(h, d_dm_out, st);
    switch (h->store) {
        case RTC_F32: return launch_dt<RTC_F32>(h, d_frame, d_dm_out, d_s_meas, head, st, fh, d_s2);
        case RTC_BF16: return launch_dt<RTC_BF16>(h, d_frame, d_dm_out, d_s_meas, head, st, fh, d_s2);
        case RTC_F16: return launch_dt<RTC_F16>(h, d_frame, d_dm_out, d_s_meas, head, st, fh, d_s2);
        case RTC_FP8_E4M3: return launch_dt<RTC_FP8_E4M3>(h, d_frame, d_dm_out, d_s_meas, head, st, fh, d_s2);
        case RTC_INT8: return launch_dt<RTC_INT8>(h, d_frame, d_dm_out, d_s_meas, head, st, fh, d_s2);
        default: return cudaErrorInvalidValue;
    }
}
