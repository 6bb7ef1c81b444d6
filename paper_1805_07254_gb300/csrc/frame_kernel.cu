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
// slice.  The block's set-up, the subaperture positions, the calibration data and, as
// plan_launch says, the first matrix tiles come before the previous kernel of the stream
// has finished; the block waits for it before it reads pixels.
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
// A small system's sum is done by the last streaming block instead (last_block_sum),
// except for HOST frames.
//
// Measured, frame after frame on one stream (one cooperative kernel with a grid barrier
// -> this): ELT FP32 28.8 -> 22.8 us (its bytes need 21.3), INT8 20.9 -> 13.0, BF16 with
// prediction 28.3 -> 24.1, six ELT sensors FP8 59.4 -> 48.0, 41x41 FP16 12.3 -> 6.8 of GPU
// time (8.8 with the two launches' host time, which bounds it) and 8x8 FP32 12.3 -> 6.1
// (7.2).

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

// LAST: the last block also sums (last_block_sum), and the launch is the whole frame.
// CHAIN: small slices (chain_rule).
template <int DT, int NPX, bool HOST, bool LAST, bool CHAIN>
__global__ void __launch_bounds__(kFrameRegThreads, 1)
frame_kernel(rtc_pixel::PixelArgs px, Args g, FrameHost fh, SumArgs sa, unsigned* ctr) {
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
    consume<DT, CHAIN>(g, pl, sh, tid, 0);
    if (LAST) {
        __shared__ int last;
        last_block_sum(sa, ctr, reinterpret_cast<float*>(smem), &last, tid);
    }
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
template <int DT, bool LAST, bool CHAIN>
__global__ void __launch_bounds__(kFrameRegThreads, 1)
frame_pred_kernel(Args g, rtc_pred::PredArgs pa, int head, SumArgs sa, unsigned* ctr) {
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
    consume<DT, CHAIN>(g, pl, sh, tid, 0);
    if (LAST) {
        __shared__ int last;
        last_block_sum(sa, ctr, reinterpret_cast<float*>(smem), &last, tid);
    }
}

template <int DT, int NPX, bool CHAIN>
cudaError_t launch_chain(const rtc_handle* h, const Launch& L, const rtc_pixel::PixelArgs& px, const Args& g,
                       const FrameHost* fh, bool last, const SumArgs& sa, cudaStream_t st) {
    const dim3 grid(L.G), block(kThreads);
    unsigned* ctr = h->d_lastctr;
    if (fh) return launch_pdl(frame_kernel<DT, NPX, true, false, CHAIN>, grid, block, L.smem, st, px, g, *fh, sa, ctr);
    if (last)
        return launch_pdl(frame_kernel<DT, NPX, false, true, CHAIN>, grid, block, L.smem, st, px, g, FrameHost{}, sa, ctr);
    return launch_pdl(frame_kernel<DT, NPX, false, false, CHAIN>, grid, block, L.smem, st, px, g, FrameHost{}, sa, ctr);
}

template <int DT, int NPX>
cudaError_t launch_npx(const rtc_handle* h, const Launch& L, const rtc_pixel::PixelArgs& px, const Args& g,
                       const FrameHost* fh, bool last, const SumArgs& sa, cudaStream_t st) {
    return L.chain ? launch_chain<DT, NPX, CanChain<DT>::v>(h, L, px, g, fh, last, sa, st)
                   : launch_chain<DT, NPX, false>(h, L, px, g, fh, last, sa, st);
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
    const bool last = !fh && last_block_sums(h->sl_S, h->cfg.nact);
    const SumArgs sa = last ? sum_args(h, d_dm_out) : SumArgs{};
    const bool n10 = h->cfg.npx == 10;
    cudaError_t e;
    if (!pred) {
        e = n10 ? launch_npx<DT, 10>(h, L, px, g, fh, last, sa, st) : launch_npx<DT, 0>(h, L, px, g, fh, last, sa, st);
    } else {
        const dim3 grid(L.G), block(kThreads);
        if (!fh) e = launch_calib_cog(h, d_frame, d_s_meas, d_s2, true, st);
        else if (n10) e = launch_pdl(frame_slopes_kernel<10>, grid, block, 0, st, px, g, *fh);
        else e = launch_pdl(frame_slopes_kernel<0>, grid, block, 0, st, px, g, *fh);
        constexpr bool kCan = CanChain<DT>::v;
        const auto k = L.chain ? (last ? frame_pred_kernel<DT, true, kCan> : frame_pred_kernel<DT, false, kCan>)
                               : (last ? frame_pred_kernel<DT, true, false> : frame_pred_kernel<DT, false, false>);
        if (e == cudaSuccess) e = launch_pdl(k, grid, block, L.smem, st, g, pred_args(h), head, sa, h->d_lastctr);
    }
    return e == cudaSuccess && !last ? launch_sum(h, d_dm_out, st, fh) : e;
}

template <typename K>
cudaError_t configure(K kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kDynSmemBudget));
}

template <int DT, int NPX, bool CHAIN>
cudaError_t configure_npx() {
    cudaError_t e = configure(frame_kernel<DT, NPX, false, false, CHAIN>);
    if (e == cudaSuccess) e = configure(frame_kernel<DT, NPX, false, true, CHAIN>);
    if (e == cudaSuccess) e = configure(frame_kernel<DT, NPX, true, false, CHAIN>);
    return e;
}

template <int DT, bool CHAIN>
cudaError_t configure_chain() {
    cudaError_t e = configure_npx<DT, 10, CHAIN>();
    if (e == cudaSuccess) e = configure_npx<DT, 0, CHAIN>();
    if (e == cudaSuccess) e = configure(frame_pred_kernel<DT, false, CHAIN>);
    if (e == cudaSuccess) e = configure(frame_pred_kernel<DT, true, CHAIN>);
    return e;
}

template <int DT>
cudaError_t configure_dt() {
    const cudaError_t e = configure_chain<DT, false>();
    return e == cudaSuccess && CanChain<DT>::v ? configure_chain<DT, CanChain<DT>::v>() : e;
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
