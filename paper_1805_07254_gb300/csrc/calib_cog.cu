// Stand-alone pixel stage: calibration, centre of gravity and slope packing for
// every valid subaperture of every WFS (Sec. 2.1, Fig. 3 (a)-(b)); a half-warp per
// subaperture, as in the fused frame kernel, which runs the same device code
// (pixel.cuh).
//
// An ELT frame is 4 MB in and 32 KB out: two dependent rounds of loads (position,
// pixels), not bandwidth.  So the stage's time in a run of frames is mostly launch and
// drain, and the launches overlap (programmatic dependent launch): a block fetches its
// subapertures' positions and calibration data, and brings their pixel lines into L2,
// while the previous kernel drains, and waits for it only before it reads pixels.  The
// slopes go straight into the caller's buffer as well as the resident one.  Measured,
// ELT, frame after frame: 2.8 us a frame on the GPU (3.0 without the lines in L2; 3.9 us
// with the caller's Python) against 10.2 us for a warp per subaperture in a plain launch
// and a device copy of the slopes after it.

#include "launch.cuh"
#include "pixel.cuh"

namespace {

constexpr int kPerBlock = kCalibThreads / 16;

// EARLY: let the successor start at once (the prediction kernel, whose set-up and matrix
// prefetch overlap this one); else after the wait: in a run of pixel stages alone,
// waiting blocks of many later frames would fill the SMs (5.5 us a frame against 3.0).
template <int NPX, bool EARLY>
__global__ void __launch_bounds__(kCalibThreads) calib_cog_kernel(rtc_pixel::PixelArgs p) {
    if (EARLY) pdl_launch_dependents();
    const int gi = blockIdx.x * kPerBlock + (threadIdx.x >> 4);
    const bool valid = gi < p.n_valid * p.n_wfs;
    const int2 pos = rtc_pixel::subap_pos(p, gi, valid);
    rtc_pixel::prefetch_rows_l2(p, gi, valid, pos, threadIdx.x);
    rtc_pixel::subap_slopes_at<NPX, rtc_pixel::kPixelL2, 16>(
        p, p.frame, p.s, gi, valid, threadIdx.x & 31, pos, rtc_pixel::NoHook(), []() {
            pdl_wait();
            if (!EARLY) pdl_launch_dependents();
        });
}

template <int NPX>
cudaError_t launch_t(const rtc_pixel::PixelArgs& p, dim3 grid, bool early, cudaStream_t st) {
    const dim3 block(kCalibThreads);
    return early ? launch_pdl(calib_cog_kernel<NPX, true>, grid, block, 0, st, p)
                 : launch_pdl(calib_cog_kernel<NPX, false>, grid, block, 0, st, p);
}

}  // namespace

rtc_pixel::PixelArgs pixel_args(const rtc_handle* h, const uint16_t* d_frame, float* d_s, float* d_s2) {
    return rtc_pixel::PixelArgs{d_frame,   h->side,      h->cfg.npx,  h->n_valid, h->cfg.n_wfs, h->d_rc,
                                h->d_dark, h->d_gainmap, h->thr_mode, h->thr,     d_s,          d_s2};
}

cudaError_t launch_calib_cog(const rtc_handle* h, const uint16_t* d_frame, float* d_s, float* d_s2, bool early,
                             cudaStream_t st) {
    const int n = h->n_valid * h->cfg.n_wfs;
    if (n == 0) return cudaSuccess;
    const dim3 grid((n + kPerBlock - 1) / kPerBlock);
    const rtc_pixel::PixelArgs p = pixel_args(h, d_frame, d_s, d_s2);
    switch (h->cfg.npx) {
        case 8: return launch_t<8>(p, grid, early, st);
        case 10: return launch_t<10>(p, grid, early, st);
        case 16: return launch_t<16>(p, grid, early, st);
        default: return launch_t<0>(p, grid, early, st);
    }
}
