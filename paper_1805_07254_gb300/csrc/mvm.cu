// Load-time storage of the control matrix in the handle's slice-major layout
// (stream_mvm.cuh).

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "rtc_internal.h"
#include "stream_mvm.cuh"

namespace {

using rtc_mvm::Esize;
using rtc_mvm::RowScaled;

// --- load-time layout ------------------------------------------------------------

// Code of x / sc in the row-scaled formats (one correctly rounded FP32 division).
template <int DT>
__device__ __forceinline__ unsigned char encode_scaled(float x, float sc) {
    const float q = __fdiv_rn(x, sc);
    if (DT == RTC_FP8_E4M3) return __nv_cvt_float_to_fp8(q, __NV_SATFINITE, __NV_E4M3);
    const int i = max(-127, min(127, __float2int_rn(q)));       // nearest, ties to even
    return static_cast<unsigned char>(static_cast<signed char>(i));
}

// Per-row scale = max |M_r| / qmax (1 for a zero row), one block per row.
template <int DT>
__global__ void row_scale_kernel(const float* __restrict__ src, int ncol, float* __restrict__ scale) {
    constexpr float qmax = DT == RTC_FP8_E4M3 ? 448.0f : 127.0f;
    __shared__ float wmax[32];
    const int row = blockIdx.x;
    const float* in = src + static_cast<size_t>(row) * ncol;
    float m = 0.f;
    for (int j = threadIdx.x; j < ncol; j += blockDim.x) m = fmaxf(m, fabsf(in[j]));
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        float mm = 0.f;
        for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) mm = fmaxf(mm, wmax[w]);
        scale[row] = mm > 0.f ? __fdiv_rn(mm, qmax) : 1.0f;
    }
}

// One row per block: FP32 column c -> its slice's row in the stored type.
template <int DT>
__global__ void layout_f32_kernel(const float* __restrict__ src, int ncol, const int2* __restrict__ colmap,
                                  const long long* __restrict__ off, const int* __restrict__ rowbytes,
                                  const float* __restrict__ scale, unsigned char* __restrict__ dst) {
    const int row = blockIdx.x;
    const float sc = RowScaled<DT>::v ? scale[row] : 1.f;
    for (int c = threadIdx.x; c < ncol; c += blockDim.x) {
        const int2 sj = colmap[c];
        unsigned char* p =
            dst + rtc_mvm::slice_elem_offset(off[sj.x], rowbytes[sj.x], row, sj.y * Esize<DT>::v, Esize<DT>::v);
        const float v = src[static_cast<size_t>(row) * ncol + c];
        if (DT == RTC_F32) *reinterpret_cast<float*>(p) = v;
        else if (DT == RTC_BF16) *reinterpret_cast<__nv_bfloat16*>(p) = __float2bfloat16_rn(v);
        else if (DT == RTC_F16) *reinterpret_cast<__half*>(p) = __float2half_rn(v);
        else *p = encode_scaled<DT>(v, sc) ^ (DT == RTC_INT8 ? rtc_mvm::kInt8Flip : 0);
    }
}

// One row per block: an element of esize bytes, already in the stored type (flip: xor of
// every byte).
__global__ void layout_raw_kernel(const unsigned char* __restrict__ src, int ncol, int esize, unsigned char flip,
                                  const int2* __restrict__ colmap, const long long* __restrict__ off,
                                  const int* __restrict__ rowbytes, unsigned char* __restrict__ dst) {
    const int row = blockIdx.x;
    for (int c = threadIdx.x; c < ncol; c += blockDim.x) {
        const int2 sj = colmap[c];
        unsigned char* p = dst + rtc_mvm::slice_elem_offset(off[sj.x], rowbytes[sj.x], row, sj.y * esize, esize);
        const unsigned char* q = src + (static_cast<size_t>(row) * ncol + c) * esize;
        for (int b = 0; b < esize; ++b) p[b] = q[b] ^ flip;
    }
}

__global__ void relayout_kernel(const unsigned char* __restrict__ src, const int2* __restrict__ src_map,
                                const long long* __restrict__ src_off, const int* __restrict__ src_rb,
                                int ncol, int esize, const int2* __restrict__ dst_map,
                                const long long* __restrict__ dst_off, const int* __restrict__ dst_rb,
                                unsigned char* __restrict__ dst) {
    const int row = blockIdx.x;
    for (int c = threadIdx.x; c < ncol; c += blockDim.x) {
        const int2 a = src_map[c], b = dst_map[c];
        const unsigned char* q =
            src + rtc_mvm::slice_elem_offset(src_off[a.x], src_rb[a.x], row, a.y * esize, esize);
        unsigned char* p =
            dst + rtc_mvm::slice_elem_offset(dst_off[b.x], dst_rb[b.x], row, b.y * esize, esize);
        for (int k = 0; k < esize; ++k) p[k] = q[k];
    }
}

}  // namespace

cudaError_t launch_layout(int src, int store, const void* d_src, int nact, int ncol,
                          const int2* d_colmap, const long long* d_off, const int* d_rowbytes,
                          float* d_scale, void* d_dst, cudaStream_t st) {
    if (nact <= 0 || ncol <= 0) return cudaSuccess;
    unsigned char* dst = static_cast<unsigned char*>(d_dst);
    if (src == store) {
        const int esize = store == RTC_F32 ? 4 : (store == RTC_BF16 || store == RTC_F16) ? 2 : 1;
        layout_raw_kernel<<<nact, 256, 0, st>>>(static_cast<const unsigned char*>(d_src), ncol, esize,
                                                store == RTC_INT8 ? rtc_mvm::kInt8Flip : 0, d_colmap, d_off, d_rowbytes, dst);
        return cudaGetLastError();
    }
    if (src != RTC_F32) return cudaErrorInvalidValue;
    const float* f = static_cast<const float*>(d_src);
    switch (store) {
        case RTC_BF16:
            layout_f32_kernel<RTC_BF16><<<nact, 256, 0, st>>>(f, ncol, d_colmap, d_off, d_rowbytes, d_scale, dst);
            break;
        case RTC_F16:
            layout_f32_kernel<RTC_F16><<<nact, 256, 0, st>>>(f, ncol, d_colmap, d_off, d_rowbytes, d_scale, dst);
            break;
        case RTC_FP8_E4M3:
            row_scale_kernel<RTC_FP8_E4M3><<<nact, 256, 0, st>>>(f, ncol, d_scale);
            layout_f32_kernel<RTC_FP8_E4M3><<<nact, 256, 0, st>>>(f, ncol, d_colmap, d_off, d_rowbytes, d_scale, dst);
            break;
        case RTC_INT8:
            row_scale_kernel<RTC_INT8><<<nact, 256, 0, st>>>(f, ncol, d_scale);
            layout_f32_kernel<RTC_INT8><<<nact, 256, 0, st>>>(f, ncol, d_colmap, d_off, d_rowbytes, d_scale, dst);
            break;
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_relayout(int esize, const void* d_old, const int2* d_old_colmap,
                            const long long* d_old_off, const int* d_old_rowbytes, int nact, int ncol,
                            const int2* d_new_colmap, const long long* d_new_off, const int* d_new_rowbytes,
                            void* d_new, cudaStream_t st) {
    if (nact <= 0 || ncol <= 0) return cudaSuccess;
    relayout_kernel<<<nact, 256, 0, st>>>(static_cast<const unsigned char*>(d_old), d_old_colmap, d_old_off,
                                          d_old_rowbytes, ncol, esize, d_new_colmap, d_new_off,
                                          d_new_rowbytes, static_cast<unsigned char*>(d_new));
    return cudaGetLastError();
}
