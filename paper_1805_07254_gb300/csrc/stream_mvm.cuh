// Device code of the reconstruction d = M s fused with the leaky integrator
// a <- leak * a + g * d (Fig. 3 (c)-(d)), shared by the stand-alone reconstruction
// kernel, the fused frame kernel and the persistent loop kernel.
//
// Decomposition (Sec. 2.3, 2.3.5).  As in the paper, where each thread takes a set
// of subapertures, multiplies the matrix columns of their slopes and leaves a
// partial DM vector that a tree then sums, the slope columns are cut into S slices
// of consecutive subapertures (S = the SM count, or the number of subapertures if
// smaller).  rtc_load_cmat stores the matrix slice by slice: slice s is one
// contiguous [nact][w_s] block, its w_s = 2 n_s columns being the slice's x slopes
// then its y slopes, each row padded to a multiple of 4 bytes.  A block of a fused
// kernel takes a run of whole slices and computes those subapertures' slopes
// itself, so its share of the product starts as soon as its own pixels are done,
// without waiting for any other block; it writes one partial vector per slice.
// Once every block is done the S partials of each row are summed in a fixed order (warp
// w sums the slices w, w+14, w+28, ... in turn for 32 consecutive rows with coalesced
// loads, then a fixed pairwise tree over the 14 warps), with the FP8/INT8 row scale
// and the integrator: by the sum kernel that follows a per-frame kernel
// (mvm_reduce_kernel), or after a grid barrier in the persistent loop.
// The result does not depend on the number of blocks or on their timing.
//
// Movement.  A slice streams in tiles of R rows, bulk asynchronous copies
// (`cp.async.bulk`) completing on a per-stage mbarrier, through a ring of up to 32
// stages in shared memory that one producer thread fills and 14 consumer warps
// drain.
//
// Arithmetic.  FP32 rows: T consecutive lanes take one row of a tile (T = 1 for
// ELT-sized slices, more when rows are long, so that at least two stages fit) and read it
// in units of 16, 8 or 4 bytes, the widest that divides the row an odd number of times
// (rows are padded until one does), so that the rows a warp reads at once fall in
// different banks; all lanes read the same units of the slice's slopes at the same
// time (shared-memory broadcasts).  1- and 2-byte stores go to the tensor cores, 16 rows
// an instruction, the slopes split into parts (see make_bfrag), or, where slices are
// small (chain_rule) or a slope does not split exactly (wide_slices), through FP32 FMAs;
// the FP8 and INT8 row scales are applied once per row after the sum over slices.
//
// Every wait is bounded (200 ms of %globaltimer); a wait that expires records
// RTC_ETIMEDOUT in the status word, the block skips the rest of its work, lets its
// copies land and returns.
#pragma once

#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <type_traits>

#include "rtc_internal.h"

namespace rtc_mvm {

constexpr int kConsumerWarps = 14;
constexpr int kConsumers = kConsumerWarps * 32;
constexpr int kThreads = kConsumers + 32;          // + one producer warp
constexpr int kMaxStages = 32;
// Smallest ring stage the launch plan aims for, in bytes (two stages of ~96 KB
// measured faster than more, smaller ones: fewer per-tile handshakes).
constexpr size_t kMinTileBytes = 96 * 1024;
constexpr size_t kMinTileBytes8 = 48 * 1024;       // of 1-byte stores (four groups of rows a warp)
// Rows of one slice's tile per consumer thread, at most (narrow slices pack several
// rows into a stage sized for the widest one).
constexpr int kMaxRowsPerThread = 32;
// Largest matrix streamed with the default L2 policy (of the 126 MB L2).
constexpr long long kL2KeepBytes = 80ll << 20;
constexpr unsigned long long kWaitNs = 200ull * 1000 * 1000;
constexpr int kMaxLocalFloats = 8192;              // slopes of a block's slices (32 KB), as slope_floats pads them
constexpr int kMaxRowFloats = 4096;                // rows a block reduces, at most
constexpr size_t kDynSmemBudget = 227 * 1024 - 2048;  // dynamic shared memory per block
// The per-frame kernels leave room on their SM for a block of the sum kernel
// (mvm_reduce_kernel: 2 KB of shared memory, 448 threads of 32 registers, so at most 104
// registers for theirs: the bound of 608 threads).
constexpr size_t kFrameSmemBudget = 223 * 1024;
constexpr int kFrameRegThreads = 608;
constexpr int kMaxSlices = 256;
constexpr int kSlicesPerWarp = (kMaxSlices + kConsumerWarps - 1) / kConsumerWarps;
constexpr uint32_t kCopyBytes = 8192;              // largest single bulk copy of a tile

template <int DT> struct Esize;
template <> struct Esize<RTC_F32> { static constexpr int v = 4; };
template <> struct Esize<RTC_BF16> { static constexpr int v = 2; };
template <> struct Esize<RTC_F16> { static constexpr int v = 2; };
template <> struct Esize<RTC_FP8_E4M3> { static constexpr int v = 1; };
template <> struct Esize<RTC_INT8> { static constexpr int v = 1; };

// Stored types whose rows carry one FP32 scale, applied once after the row's sum.
template <int DT> struct RowScaled { static constexpr bool v = DT == RTC_FP8_E4M3 || DT == RTC_INT8; };

// ---- PTX wrappers -------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bulk copy global -> shared completing on an mbarrier, with an L2 eviction policy.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes,
                                         uint32_t bar, unsigned long long policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1], %2, [%3], %4;"
        ::"r"(dst), "l"(src), "r"(bytes), "r"(bar), "l"(policy)
        : "memory");
}
// L2 policies for the matrix stream.  A matrix larger than L2 goes through without
// displacing the calibration maps, frames and partial vectors (evict_first); one
// that fits beside them keeps the default policy, so that frame after frame it can
// stay in L2.
enum L2Policy { kL2Normal = 0, kL2Stream = 1 };
__device__ __forceinline__ unsigned long long matrix_policy(int mode) {
    unsigned long long p;
    if (mode == kL2Stream)
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    else
        asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}
// Bulk prefetch of global bytes into L2 (no shared memory, no completion).
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t addr) {
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t addr) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(addr));
    return v;
}

// Access unit of a slice row of rb bytes: the widest of 16, 8, 4 bytes that divides
// the row an odd number of times, so that the rows a warp reads at once (rb bytes
// apart) fall in different banks.  rtc_load_cmat pads rows until one exists.
__host__ __device__ __forceinline__ int row_unit(int rb) {
    if (rb % 16 == 0 && (rb / 16) % 2 == 1) return 16;
    if (rb % 8 == 0 && (rb / 8) % 2 == 1) return 8;
    if (rb % 4 == 0 && (rb / 4) % 2 == 1) return 4;
    return 0;
}
// Bytes of a slice's row of 2 n entries until an access unit exists, and the floats of its
// slopes.  (Fragment-order slices are neither padded so, nor their slopes; the limit on
// a block's slopes counts every store alike.)
inline int row_bytes(int n, int esz) {
    int rb = (2 * n * esz + 3) / 4 * 4;
    while (row_unit(rb) == 0) rb += 4;
    return rb;
}
inline int slope_floats(int n, int esz) { return (row_bytes(n, esz) / esz + 3) / 4 * 4; }
// A handle's INT8 codes are stored with the sign bit flipped (code + 128 as an unsigned
// byte), which widen4 wants.
constexpr unsigned char kInt8Flip = 0x80;

// Byte offset of element byte cb of row `row` of a slice at byte off, rb bytes per row,
// es bytes per element.  FP32 slices (es 4) are row-major.  The 1- and 2-byte stores
// are in fragment order: rows in groups of 16 (16 rb bytes each, the last one padded with
// zero rows), and within a group
//   - 1-byte: the columns' first whole 32s, 512 bytes each: for lane (g, t) = (row % 8,
//     column / 8) 16 bytes, 8 columns of row g then the same 8 of row g + 8;
//   - the next whole 16s (2-byte: all of them), 256 es bytes each: for lane (row % 8,
//     column / 4) 4 columns of row g then the same 4 of row g + 8;
//   - the next whole 8, 128 es bytes: for lane (row % 8, column / 2) 2 columns of row g,
//     then of row g + 8;
//   - the last 2, 4 or 6 columns, the same for as many quarters t as there are pairs.
// So a lane of a warp reads its share of an mma.m16n8k16 A operand, of two, or of half a
// one as one vector, and the warp's read is consecutive bytes.
__host__ __device__ __forceinline__ size_t slice_elem_offset(long long off, int rb, int row, int cb, int es) {
    if (es == 4) return static_cast<size_t>(off) + static_cast<size_t>(row) * rb + cb;
    const int r = row & 15, K = rb / es, b = cb % es;
    int c = cb / es;
    size_t at = static_cast<size_t>(off) + static_cast<size_t>(row >> 4) * 16 * rb;
    const int k32 = es == 1 ? K & ~31 : 0;
    if (c < k32) return at + (c >> 5) * 512 + ((r & 7) * 4 + ((c & 31) >> 3)) * 16 + (r >> 3) * 8 + (c & 7);
    at += static_cast<size_t>(k32) * 16;
    c -= k32;
    const int k16 = (K - k32) & ~15;
    if (c < k16)
        return at + ((c >> 4) * 256 + ((r & 7) * 4 + ((c & 15) >> 2)) * 8 + (r >> 3) * 4 + (c & 3)) * es + b;
    at += static_cast<size_t>(k16) * 16 * es;
    c -= k16;
    const int left = (K - k32 - k16), k8 = left & 8;
    if (c < k8) return at + ((r & 7) * 8 + (c >> 1) * 2) * 2 * es + ((r >> 3) * 2 + (c & 1)) * es + b;
    at += k8 * 16 * es;
    c -= k8;
    return at + ((r & 7) * (left - k8) + (c >> 1) * 2) * 2 * es + ((r >> 3) * 2 + (c & 1)) * es + b;
}

__device__ __forceinline__ void consumer_sync() {          // all consumer warps
    asm volatile("bar.sync 1, %0;" ::"n"(kConsumers) : "memory");
}

// Bounded wait on an mbarrier phase; false if it expired or (when abort is given)
// the block aborted.
__device__ __forceinline__ bool wait_phase(uint32_t bar, uint32_t parity, volatile int* abort) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (abort && *abort) return false;
        if (global_ns() - t0 > kWaitNs) return false;
    }
}

// ---- widening dot products: acc += <one 4-byte word of a row, its slopes> -------
__device__ __forceinline__ float2 e4m3x2_to_float2(uint32_t two) {
    __half2_raw hr = __nv_cvt_fp8x2_to_halfraw2(static_cast<__nv_fp8x2_storage_t>(two), __NV_E4M3);
    return __half22float2(*reinterpret_cast<__half2*>(&hr));
}

// Four signed 8-bit codes (bias-flipped by xor 0x80) -> exact floats: the byte
// goes into the low mantissa bits of 2^23, so the float is 2^23 + code + 128.
__device__ __forceinline__ float i8_to_float(uint32_t flipped, int k) {
    return __uint_as_float(__byte_perm(flipped, 0x4B000000u, 0x7650 + k)) - 8388736.0f;
}

// acc += <word w, its EPW slopes s>.  (Placing FP8 / FP16 bits at the top of an FP32
// mantissa and pre-scaling the slopes by 2^120 / 2^112 avoids the conversion
// instructions but measured slower than the hardware conversions.)
template <int DT>
__device__ __forceinline__ float word_dot(float acc, uint32_t w, const float* s) {
    if (DT == RTC_F32) {
        acc = fmaf(__uint_as_float(w), s[0], acc);
    } else if (DT == RTC_BF16) {
        acc = fmaf(__uint_as_float(w << 16), s[0], acc);
        acc = fmaf(__uint_as_float(w & 0xffff0000u), s[1], acc);
    } else if (DT == RTC_F16) {
        __half2_raw hr;
        hr.x = static_cast<unsigned short>(w & 0xffffu);
        hr.y = static_cast<unsigned short>(w >> 16);
        const float2 f = __half22float2(*reinterpret_cast<__half2*>(&hr));
        acc = fmaf(f.x, s[0], acc);
        acc = fmaf(f.y, s[1], acc);
    } else if (DT == RTC_FP8_E4M3) {
        const float2 a = e4m3x2_to_float2(w & 0xffffu);
        const float2 b = e4m3x2_to_float2(w >> 16);
        acc = fmaf(a.x, s[0], acc);
        acc = fmaf(a.y, s[1], acc);
        acc = fmaf(b.x, s[2], acc);
        acc = fmaf(b.y, s[3], acc);
    } else {
        const uint32_t x = w ^ 0x80808080u;
        acc = fmaf(i8_to_float(x, 0), s[0], acc);
        acc = fmaf(i8_to_float(x, 1), s[1], acc);
        acc = fmaf(i8_to_float(x, 2), s[2], acc);
        acc = fmaf(i8_to_float(x, 3), s[3], acc);
    }
    return acc;
}

// Integrator update of one actuator from its previous state and row scale.
template <int DT>
__device__ __forceinline__ float integrate_row(int row, float d, float a_prev, float sc,
                                               float* __restrict__ a, float* __restrict__ dm_out,
                                               float gain, float leak) {
    if (RowScaled<DT>::v) d *= sc;
    const float an = fmaf(leak, a_prev, gain * d);
    a[row] = an;
    if (dm_out) dm_out[row] = an;
    return an;
}

// ---- plan ----------------------------------------------------------------------

// The slice table of a loaded matrix (device arrays).
struct Slices {
    const long long* off;    // [S] byte offset of slice s in the matrix (16-byte aligned)
    const int* rowbytes;     // [S] bytes per row of slice s (multiple of 4)
    const int* g0;           // [S + 1] first subaperture (w * n_valid + i) of slice s
    const int* loc;          // [S + 1] float offset of slice s's slopes in a local vector
    int S;
    int nt;                  // subapertures over all WFS
    int equal;               // g0[s] = nt s / S (the default cut): computed, not loaded
};

struct Args {
    const unsigned char* M;  // slice-major matrix
    Slices sl;
    int nact, n_valid;       // rows; valid subapertures per WFS
    int T, R;                // lanes per row, rows per tile (T * R = kConsumers)
    int stage_bytes, nst;    // the ring: nst stages of stage_bytes (R rows of the widest slice)
    int l2_policy;           // L2Policy of the matrix stream
    int region;              // shared scratch bytes of a fused phase (before the slopes)
    int loc_floats;          // floats of the largest block-local slope vector
    int row_floats;          // rows a block reduces, at most
    int frag;                // slices in fragment order (1- and 2-byte stores; see slice_elem_offset)
    int pre_tiles;           // tiles requested before the previous kernel is complete
    int l2_ahead;            // tiles brought into L2 once the ring has been requested
    int max_slices;          // slices of a block, at most
    int bf_floats;           // floats of a block's B fragments (0 for FP32)
    const float* s;          // stand-alone reconstruction: the full slope vector (else unused)
    const float* scale;      // [nact] row scales (FP8, INT8)
    float* partial;          // [S][pstride] partial DM vectors
    int pstride;             // nact, rounded up to the groups of 16 rows
    float* a;                // [nact] integrator state
    float gain, leak;
    int* status;             // device error word, kept until the host reads it
    int* cut;                // mark of this launch alone (see record_timeout)
};

struct Shared {
    unsigned long long full_bar[kMaxStages];
    unsigned long long empty_bar[kMaxStages];
    volatile int abort_flag;
};

// What one block does.
struct Plan {
    int sb0, sb1;            // slices [sb0, sb1)
    int g0, g1;              // subapertures [g0, g1)
    int r0, r1;              // rows the block reduces
    int rb0, n0, loc0;       // first slice: bytes per row, subapertures, local offset
    uint32_t ring;           // shared address of the ring
    unsigned char* scratch;  // fused-phase scratch (region bytes)
    float* loc;              // block-local slopes: each slice's x then y block, zero padded
    float* bf;               // fragment-order slices: their B fragments (make_bfrag)
    float* bscale;           // and what each slice's products are scaled back by
    float* a_pre;            // [r1 - r0] integrator state of the rows the block reduces
    float* sc_pre;           // [r1 - r0] their row scales
    float* red;              // [kConsumerWarps][32] warp sums of the sum over slices
};

__device__ __forceinline__ void init_shared(Shared& sh) {
    for (int i = 0; i < kMaxStages; ++i) {
        mbar_init(smem_addr(&sh.full_bar[i]), 1);
        mbar_init(smem_addr(&sh.empty_bar[i]), kConsumerWarps);
    }
    sh.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ Plan make_plan(const Args& g, unsigned char* smem) {
    Plan pl;
    const unsigned S = g.sl.S;
    // (32-bit products: a plan has at most 256 slices, and at most 4096 subapertures a slice
    // and rows a block; a 64-bit division is some 80 instructions in every warp)
    const unsigned b = blockIdx.x, G = gridDim.x;
    pl.sb0 = S * b / G;
    pl.sb1 = S * (b + 1) / G;
    // the block's subapertures: with the default cut computed, so that the pixel
    // stage does not wait for a table load before it can fetch positions
    if (g.sl.equal) {
        const unsigned nt = g.sl.nt;
        pl.g0 = nt * pl.sb0 / S;
        pl.g1 = nt * pl.sb1 / S;
        pl.n0 = nt * (pl.sb0 + 1) / S - pl.g0;
    } else {
        pl.g0 = g.sl.g0[pl.sb0];
        pl.g1 = g.sl.g0[pl.sb1];
        pl.n0 = g.sl.g0[pl.sb0 + 1] - pl.g0;
    }
    // the first slice's layout, read once here rather than on the frame's critical path
    pl.rb0 = g.sl.rowbytes[pl.sb0];
    pl.loc0 = g.sl.loc[pl.sb0];
    pl.r0 = static_cast<unsigned>(g.nact) * b / G;
    pl.r1 = static_cast<unsigned>(g.nact) * (b + 1) / G;
    const int ring_bytes = g.nst * g.stage_bytes;
    pl.ring = smem_addr(smem);
    pl.scratch = smem + ring_bytes;
    pl.loc = reinterpret_cast<float*>(smem + ring_bytes + g.region);
    pl.bf = pl.loc + g.loc_floats;
    pl.bscale = pl.bf + g.bf_floats;
    pl.a_pre = pl.bscale + (g.frag ? g.max_slices : 0);
    pl.sc_pre = pl.a_pre + g.row_floats;
    pl.red = pl.sc_pre + g.row_floats;
    return pl;
}

// Where subaperture gi (one of the block's) puts its x and y slopes in the
// block-local vector.
__device__ __forceinline__ void local_index(const Args& g, const Plan& pl, int gi, int& ix, int& iy) {
    if (gi < pl.g0 + pl.n0) {           // the first slice
        ix = gi - pl.g0;
        iy = ix + pl.n0;
        return;
    }
    int s = pl.sb0 + 1;
    while (s + 1 < pl.sb1 && g.sl.g0[s + 1] <= gi) ++s;
    const int base = g.sl.loc[s] - pl.loc0;
    const int n = g.sl.g0[s + 1] - g.sl.g0[s];
    ix = base + (gi - g.sl.g0[s]);
    iy = ix + n;
}

// Consumers: clear the block-local slope vector (its padding stays zero).
__device__ __forceinline__ void clear_local(const Args& g, const Plan& pl, int tid) {
    for (int i = tid; i < g.loc_floats; i += kConsumers) pl.loc[i] = 0.f;
}

// Consumers: the block's slopes from a full slope vector s (x block then y block per
// WFS).  fresh: s was written by other blocks of the same kernel (read from L2).
__device__ __forceinline__ void gather_local(const Args& g, const Plan& pl, int tid,
                                             const float* __restrict__ s, bool fresh) {
    for (int gi = pl.g0 + tid; gi < pl.g1; gi += kConsumers) {
        const int w = gi / g.n_valid, i = gi - w * g.n_valid;
        const size_t bx = static_cast<size_t>(w) * 2 * g.n_valid + i;
        int ix, iy;
        local_index(g, pl, gi, ix, iy);
        pl.loc[ix] = fresh ? __ldcg(s + bx) : __ldg(s + bx);
        pl.loc[iy] = fresh ? __ldcg(s + bx + g.n_valid) : __ldg(s + bx + g.n_valid);
    }
}

// 4-byte global -> shared copy that does not hold up the issuing thread.
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// Consumers: integrator state and row scales of the rows the block reduces, as
// asynchronous copies, so that the block's first tiles need not wait for them (a
// cold load here held every frame's stream back by about a round trip).  The
// copies are complete once rows_landed() and a consumer barrier have followed.
template <int DT>
__device__ __forceinline__ void prefetch_rows(const Args& g, const Plan& pl, int tid) {
    for (int r = pl.r0 + tid; r < pl.r1; r += kConsumers) {
        cp_async4(pl.a_pre + (r - pl.r0), g.a + r);
        if (RowScaled<DT>::v) cp_async4(pl.sc_pre + (r - pl.r0), g.scale + r);
        else pl.sc_pre[r - pl.r0] = 1.f;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// The calling thread's prefetch_rows copies have landed.  Every consumer calls it
// before the barrier that precedes reduce_rows, aborted or not (no copy may still
// be writing shared memory when the block exits).
__device__ __forceinline__ void rows_landed() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// A bounded wait of this launch expired.  The error word stays set until the host reads
// it; the mark tells the sum of this launch that partials are missing, which then leaves
// the integrator as it was and clears the mark, so that the next frame runs as usual.
__device__ __forceinline__ void record_timeout(const Args& g) {
    atomicExch(g.status, RTC_ETIMEDOUT);
    atomicExch(g.cut, RTC_ETIMEDOUT);
}

// Rows of slice tiles with rb bytes per row: R rows for the widest slice, a multiple
// of R that still fits in a stage for narrower ones.  A row is always summed by
// the same T lanes, so the tile height does not change any result.
__device__ __forceinline__ int tile_rows(const Args& g, int rb) {
    const int m = g.stage_bytes / (g.R * rb);
    return g.R * (m < 1 ? 1 : m > kMaxRowsPerThread ? kMaxRowsPerThread : m);
}

// One producer thread: stream the block's slices tile by tile into the ring.
// tl0: the running tile count at entry (barrier phases continue across calls, e.g.
// frame after frame in a persistent kernel); returns the count at exit.  drain: wait
// for the last copies to land before returning (a block must not exit with copies
// in flight).  The ring fills before the block's slopes are known and then waits for
// its consumers.  A per-frame kernel requests its first pre_tiles tiles before its
// predecessor is complete, the others after (the persistent loop has no predecessor),
// and l2_ahead further ones into L2 (see Launch::pre_tiles).  pre_tiles is at most the
// ring's stages: the bounded wait for a stage starts after the unbounded one for the
// predecessor, whose run time is not this kernel's.
__device__ __forceinline__ int produce(const Args& g, const Plan& pl, Shared& sh, int tl0 = 0, bool drain = true) {
    int tl = tl0;
    bool ok = true;
    const unsigned long long policy = matrix_policy(g.l2_policy);
    for (int s = pl.sb0; s < pl.sb1 && ok; ++s) {
        const unsigned char* base = g.M + g.sl.off[s];
        const int rb = g.sl.rowbytes[s];
        const int tr = tile_rows(g, rb);
        for (int row0 = 0; row0 < g.nact; row0 += tr, ++tl) {
            if (tl == g.pre_tiles) asm volatile("griddepcontrol.wait;" ::: "memory");
            if (g.l2_ahead && tl == g.nst) {
                const uint32_t ahead = (static_cast<uint32_t>(min(g.l2_ahead * tr, g.nact - row0)) * rb) & ~15u;
                const unsigned char* next = base + static_cast<size_t>(row0) * rb;
                for (uint32_t o = 0; o < ahead; o += kCopyBytes) bulk_prefetch_l2(next + o, min(kCopyBytes, ahead - o));
            }
            const int st = tl % g.nst;
            const int use = tl / g.nst;
            if (use > 0 && !wait_phase(smem_addr(&sh.empty_bar[st]), (use - 1) & 1, &sh.abort_flag)) {
                ok = false;
                break;
            }
            // a slice in fragment order is padded to groups of 16 rows, a row-major one to
            // 16 bytes; the tile goes as several copies
            const int left = min(tr, g.nact - row0), rows = g.frag ? (left + 15) & ~15 : left;
            const uint32_t bytes = (static_cast<uint32_t>(rows) * rb + 15u) & ~15u;
            const uint32_t fb = smem_addr(&sh.full_bar[st]);
            mbar_expect_tx(fb, bytes);
            const unsigned char* src = base + static_cast<size_t>(row0) * rb;
            for (uint32_t o = 0; o < bytes; o += kCopyBytes)
                bulk_g2s(pl.ring + st * g.stage_bytes + o, src + o, min(kCopyBytes, bytes - o), fb, policy);
        }
    }
    if (!ok && !sh.abort_flag) {
        record_timeout(g);
        sh.abort_flag = 1;
    }
    if (drain || !ok)
        for (int t = max(tl0, tl - g.nst); t < tl; ++t)
            wait_phase(smem_addr(&sh.full_bar[t % g.nst]), (t / g.nst) & 1, nullptr);
    return tl;
}

// The EPU slopes of one unit into registers with vector loads (shared-memory
// broadcasts: every lane of the warp reads the same unit at the same time).
template <int EPU>
__device__ __forceinline__ void load_unit(const float* s, float* r) {
    if constexpr (EPU % 4 == 0) {
#pragma unroll
        for (int j = 0; j < EPU; j += 4) {
            const float4 v = *reinterpret_cast<const float4*>(s + j);
            r[j] = v.x;
            r[j + 1] = v.y;
            r[j + 2] = v.z;
            r[j + 3] = v.w;
        }
    } else if constexpr (EPU == 2) {
        const float2 v = *reinterpret_cast<const float2*>(s);
        r[0] = v.x;
        r[1] = v.y;
    } else {
        r[0] = s[0];
    }
}

// acc += <one U-byte unit of a row at shared address a, its slopes r>, word by word.
template <int DT, int U>
__device__ __forceinline__ float unit_dot(float acc, uint32_t a, const float* r) {
    constexpr int EPW = 4 / Esize<DT>::v;                    // elements per 4-byte word
    if constexpr (U == 16) {
        const uint4 m = lds128(a);
        acc = word_dot<DT>(acc, m.x, r);
        acc = word_dot<DT>(acc, m.y, r + EPW);
        acc = word_dot<DT>(acc, m.z, r + 2 * EPW);
        acc = word_dot<DT>(acc, m.w, r + 3 * EPW);
    } else if constexpr (U == 8) {
        const uint2 m = lds64(a);
        acc = word_dot<DT>(acc, m.x, r);
        acc = word_dot<DT>(acc, m.y, r + EPW);
    } else {
        acc = word_dot<DT>(acc, lds32(a), r);
    }
    return acc;
}

// Slope floats a consumer lane keeps in registers for one slice.
constexpr int kSlopeRegs = 16;
// Units of a row a lane can hold the slopes of: kSlopeRegs / (elements per unit).
template <int DT, int U>
struct LaneUnits {
    static constexpr int v = kSlopeRegs * Esize<DT>::v / U > 0 ? kSlopeRegs * Esize<DT>::v / U : 1;
};

// The tiles of one slice (rb bytes per row, its slopes at pl.loc + lo); returns the
// running tile count.  Lane `part` of a row's T lanes takes the row's units part,
// part + T, ..., in that order, and the T partial sums meet in an xor butterfly.
// When a lane's units fit (LaneUnits), their slopes stay in registers for the
// whole slice and the tile is read once; otherwise every unit's slopes come from
// shared memory.  Both ways add the same terms in the same order.
template <int DT, int U>
__device__ __forceinline__ int consume_slice(const Args& g, const Plan& pl, Shared& sh, int tid,
                                             int tile, int s, int rb, int lo) {
    constexpr int EPU = U / Esize<DT>::v;                    // elements per unit
    constexpr int JM = LaneUnits<DT, U>::v;
    // launch constants in registers for the row loops
    const int T = g.T, R = g.R, nact = g.nact, nst = g.nst, stage_bytes = g.stage_bytes;
    const int lane = tid & 31;
    const int rt = tid / T;                                  // row of the tile
    const int part = tid - rt * T;                           // lane within the row's group
    const int nunits = rb / U;
    const float* sv = pl.loc + lo;
    float* out = g.partial + static_cast<size_t>(s) * g.pstride;
    const int tr = tile_rows(g, rb);
    const bool in_regs = (nunits + T - 1) / T <= JM;     // the same for the whole block
    float sr[JM][EPU];
#pragma unroll
    for (int j = 0; j < JM; ++j) {
        const int k = part + j * T;
        if (in_regs && k < nunits) {
            load_unit<EPU>(sv + k * EPU, sr[j]);
        } else {
#pragma unroll
            for (int e = 0; e < EPU; ++e) sr[j][e] = 0.f;
        }
    }
    for (int row0 = 0; row0 < nact; row0 += tr, ++tile) {
        const int st = tile % nst;
        const bool ok = __all_sync(0xffffffffu, wait_phase(smem_addr(&sh.full_bar[st]),
                                                            (tile / nst) & 1, &sh.abort_flag));
        if (!ok) {
            if (lane == 0 && !sh.abort_flag) {
                record_timeout(g);
                sh.abort_flag = 1;
            }
            continue;     // skip the work but keep reaching the block's barriers
        }
        const uint32_t stage = pl.ring + st * stage_bytes;
        // rows of this tile per lane group: the same count on every lane
        const int iters = (min(tr, nact - row0) + R - 1) / R;
        if (in_regs) {
            int i = 0;
            for (; i + 2 <= iters; i += 2) {                 // two rows in flight
                const int ra = rt + i * R, rbw = ra + R;
                const bool va = row0 + ra < nact, vb = row0 + rbw < nact;
                float acc0 = 0.f, acc1 = 0.f;
#pragma unroll
                for (int j = 0; j < JM; ++j) {
                    const int k = part + j * T;
                    if (k < nunits) {
                        if (va) acc0 = unit_dot<DT, U>(acc0, stage + ra * rb + k * U, sr[j]);
                        if (vb) acc1 = unit_dot<DT, U>(acc1, stage + rbw * rb + k * U, sr[j]);
                    }
                }
                for (int off = T >> 1; off > 0; off >>= 1) {
                    acc0 += __shfl_xor_sync(0xffffffffu, acc0, off);
                    acc1 += __shfl_xor_sync(0xffffffffu, acc1, off);
                }
                if (part == 0 && va) out[row0 + ra] = acc0;
                if (part == 0 && vb) out[row0 + rbw] = acc1;
            }
            if (i < iters) {
                const int ra = rt + i * R;
                const bool va = row0 + ra < nact;
                float acc0 = 0.f;
#pragma unroll
                for (int j = 0; j < JM; ++j) {
                    const int k = part + j * T;
                    if (k < nunits && va) acc0 = unit_dot<DT, U>(acc0, stage + ra * rb + k * U, sr[j]);
                }
                for (int off = T >> 1; off > 0; off >>= 1) acc0 += __shfl_xor_sync(0xffffffffu, acc0, off);
                if (part == 0 && va) out[row0 + ra] = acc0;
            }
        } else {
            for (int i = 0; i < iters; ++i) {
                const int ra = rt + i * R;
                const bool va = row0 + ra < nact;
                float acc = 0.f;
                if (va) {
#pragma unroll 4
                    for (int k = part; k < nunits; k += T) {
                        float r[EPU];
                        load_unit<EPU>(sv + k * EPU, r);
                        acc = unit_dot<DT, U>(acc, stage + ra * rb + k * U, r);
                    }
                }
                for (int off = T >> 1; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
                if (part == 0 && va) out[row0 + ra] = acc;
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_addr(&sh.empty_bar[st]));
    }
    return tile;
}

// ---- 1- and 2-byte stores on the tensor cores -------------------------------------
//
// A multiply-add per matrix byte or two, with the conversion to FP32 and the slope's read,
// kept the CUDA cores busy longer than the HBM takes to deliver the bytes (ELT INT8: 8.2
// us against 5.2).  mma.sync.m16n8k16 takes the matrix as its A operand in the stored
// type (BF16, FP16) or as the exactly equal FP16 values (E4M3 by the hardware
// conversion, INT8 through the mantissa of 1024), 16 rows x 16 slopes an instruction.
// The FP32 slopes are its B operand, each split exactly into three 16-bit parts in three
// of the 8 columns:
//   - BF16: the upper 8 bits of the significand, the next 8, the last 8 (truncating
//     splits: nothing overflows, and the range is FP32's own);
//   - FP16: 11 bits, 11 and 2, the second and third scaled by 2^11 and 2^22, after a
//     power of two per slice that brings the slice's largest slope just below 2^15.
// The split loses bits of slopes below 2^-37 of the slice's largest (FP16), where FP16's
// subnormals end, or below 2^-102 (BF16).  A slice that holds such a slope is marked and
// its rows are summed once more as FP32 chains (wide_slices): a matrix may well be zero
// where a dead subaperture's slope is huge.
// Products are exact and accumulate in FP32, and the three column sums meet at the end.
// Infinite and NaN slopes go whole into the first part, and an infinite sum of first
// parts (an infinite slope or matrix entry) is the row's sum.  Against 64 bits the commands
// are as near as the FP32 chains' were or nearer (relative 2-norm: ELT FP16 41x41 1.2e-7
// against 1.3e-7, six sensors FP8 2.3e-7 against 2.5e-7, BF16 loop 1.7e-7 against 2.1e-7).
// Measured, frame after frame, with FP32 chains -> so: ELT INT8 17.0 -> 13.7 us, six
// sensors FP8 54.6 -> 47.0, BF16 with prediction 26.9 -> 24.7; the persistent loop with
// the BF16 matrix in L2 23.2 -> 18.1 us a frame.
// (The 1-byte forms of mma.sync, with the slopes as E4M3 or integer digits in 8 columns,
// were no faster: the E4M3 one issues the FP16 instructions and conversions, and the
// integer one is slow on this GPU, 18.7 us for the ELT INT8 frame against 14.7.)

template <int DT> struct HalfKind { static constexpr bool v = DT != RTC_BF16; };   // FP16 operands

__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y));
}
template <int DT>
__device__ __forceinline__ void mma_dt(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint2 b) {
    if (HalfKind<DT>::v) mma_f16(c, a0, a1, a2, a3, b);
    else mma_bf16(c, a0, a1, a2, a3, b);
}

// Four 1-byte codes as two pairs of FP16 values.
template <int DT>
__device__ __forceinline__ void widen4(uint32_t w, uint32_t& lo, uint32_t& hi) {
    if (DT == RTC_FP8_E4M3) {
        asm("{\n\t.reg .b16 a, b;\n\t"
            "mov.b32 {a, b}, %2;\n\t"
            "cvt.rn.f16x2.e4m3x2 %0, a;\n\t"
            "cvt.rn.f16x2.e4m3x2 %1, b;\n\t}"
            : "=r"(lo), "=r"(hi)
            : "r"(w));
    } else {
        // stored as code + 128 (kInt8Flip): 1024 + it as FP16, minus 1152: exact
        const __half2 k = __half2half2(__ushort_as_half(0x6480));
        const uint32_t p = __byte_perm(w, 0x64646464u, 0x4140), q = __byte_perm(w, 0x64646464u, 0x4342);
        const __half2 a = __hsub2(*reinterpret_cast<const __half2*>(&p), k);
        const __half2 b = __hsub2(*reinterpret_cast<const __half2*>(&q), k);
        lo = *reinterpret_cast<const uint32_t*>(&a);
        hi = *reinterpret_cast<const uint32_t*>(&b);
    }
}

// Floats the B fragments of n slopes (a multiple of 16) take: 96 bytes a step of 16.
__host__ __device__ __forceinline__ int bfrag_floats(int n) { return n / 16 * 24; }

// Power of two that brings the largest finite of K slopes into [2^14, 2^15), and its
// inverse.  By a whole warp.
__device__ __forceinline__ void slope_scale(const float* sv, int K, int lane, float& up, float& down) {
    unsigned m = 0;                                          // largest finite magnitude, as bits
    for (int c = lane; c < K; c += 32) {
        const unsigned u = __float_as_uint(sv[c]) & 0x7fffffffu;
        if (u < 0x7f800000u) m = max(m, u);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    const int e = m ? max(static_cast<int>(m >> 23) - 127, -100) : 14;
    up = __uint_as_float(static_cast<unsigned>(127 + 14 - e) << 23);
    down = __uint_as_float(static_cast<unsigned>(127 - 14 + e) << 23);
}

// The parts of column c of a slice of K columns into its B fragments: the step, quarter
// t and place j of the matrix elements the lanes hold (slice_elem_offset's column order).
// Returns whether they may not hold all of v.
template <int DT>
__device__ __forceinline__ bool put_parts(float* frag, int K, int c, float v, float up) {
    const bool finite = (__float_as_uint(v) & 0x7f800000u) != 0x7f800000u;
    const int k32 = Esize<DT>::v == 1 ? K & ~31 : 0, rest = c - (K & ~15);
    int step = c >> 4, t = (c & 15) >> 2, j = c & 3;
    if (c < k32) {
        step = 2 * (c >> 5) + ((c & 7) >> 2);
        t = (c & 31) >> 3;
    } else if (rest >= 0) {                                  // the last, partial 16: 8, then pairs
        const int k8 = K & 8, second = rest >= k8;
        t = (rest - (second ? k8 : 0)) >> 1;
        j = 2 * second + (c & 1);
    }
    unsigned short* out = reinterpret_cast<unsigned short*>(frag) + step * 48 + t * 4 + j;
    float r = HalfKind<DT>::v ? v * up : v;
    const bool lost = v != 0.f && fabsf(r) < (HalfKind<DT>::v ? 0x1p-23f : 0x1p-102f);
#pragma unroll
    for (int n = 0; n < 3; ++n) {
        unsigned short d;
        if (HalfKind<DT>::v) {
            const __half h = __float2half_rz(r);
            d = __half_as_ushort(h);
            r = finite ? (r - __half2float(h)) * 2048.f : 0.f;
        } else {
            const unsigned u = __float_as_uint(r) & 0xffff0000u;
            d = static_cast<unsigned short>(u >> 16);
            if (n == 0 && v != v) d = 0x7fc0;                // a NaN whatever its payload
            r = finite ? r - __uint_as_float(u) : 0.f;
        }
        out[n * 16] = d;
    }
    return lost;
}

// B fragments of the block's slices from its local slopes, and what each slice's sums
// are scaled back by.  A block's only slice is shared by all its warps, several go a
// warp each.  Between consumer barriers.
template <int DT>
__device__ __forceinline__ void make_bfrag(const Args& g, const Plan& pl, int tid) {
    const int lane = tid & 31, warp = tid >> 5;
    const bool one = pl.sb1 - pl.sb0 == 1;
    for (int s = pl.sb0 + (one ? 0 : warp); s < pl.sb1; s += one ? 1 : kConsumerWarps) {
        const int rb = s == pl.sb0 ? pl.rb0 : __ldg(g.sl.rowbytes + s);
        const int lo = s == pl.sb0 ? 0 : __ldg(g.sl.loc + s) - pl.loc0;
        const int K = rb / Esize<DT>::v;
        const float* sv = pl.loc + lo;
        float* frag = pl.bf + bfrag_floats(lo);
        float up = 1.f, down = 1.f;
        if (HalfKind<DT>::v) slope_scale(sv, K, lane, up, down);
        if (lane == 0 && (!one || warp == 0)) pl.bscale[s - pl.sb0] = down;
        // the last step's places, of which the columns may leave some
        if (K & 15) {
            float* last = frag + bfrag_floats(K & ~15);
            for (int i = one ? tid : lane; i < bfrag_floats(16); i += one ? kConsumers : 32) last[i] = 0.f;
        }
        if (one) consumer_sync();
        else __syncwarp();
        bool lost = false;
        for (int c = one ? tid : lane; c < K; c += one ? kConsumers : 32) lost |= put_parts<DT>(frag, K, c, sv[c], up);
        if (lost) pl.bscale[s - pl.sb0] = 0.f;               // the mark of a slice for wide_slices
    }
}

// A slice's B fragments of a step, for the calling lane: the 12 lanes of the three parts
// hold slopes, the others zeros.
__device__ __forceinline__ uint2 bfrag(const float* frag, int step, int lane) {
    uint2 b = make_uint2(0u, 0u);
    if (lane < 12) b = reinterpret_cast<const uint2*>(frag)[step * 12 + lane];
    return b;
}

// The B fragments of a slice of at most 64 columns, kept in registers for the whole
// slice: the full steps, then the partial one.
struct SliceB {
    uint2 full[4], last;
};

// NG groups of 16 rows, group i at shared address at + i * gap: the rows' sums on each
// quad's first lane, v[group][row half].  SMALL: at most 64 columns, their B fragments in
// sb; else read step by step, once for all groups.  The groups' chains of products
// are independent.
template <int DT, int NG, bool SMALL>
__device__ __forceinline__ void frag_dot(uint32_t at, uint32_t gap, int K, int lane, const SliceB& sb,
                                         const float* frag, float (&v)[NG][2]) {
    constexpr int ES = Esize<DT>::v;
    float acc[NG][4];
#pragma unroll
    for (int i = 0; i < NG; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
    const uint32_t a16 = at + lane * 16;
    const int q16 = K >> 4;                                  // whole steps of 16
    if constexpr (ES == 1) {
        const int q32 = K >> 5;
        auto chunk = [&](int c, uint2 b0, uint2 b1) {        // 32 columns
            uint4 m[NG];
#pragma unroll
            for (int i = 0; i < NG; ++i) m[i] = lds128(a16 + i * gap + c * 512);
#pragma unroll
            for (int i = 0; i < NG; ++i) {
                uint32_t x0, x1, y0, y1, z0, z1, w0, w1;
                widen4<DT>(m[i].x, x0, x1);
                widen4<DT>(m[i].z, z0, z1);
                mma_dt<DT>(acc[i], x0, z0, x1, z1, b0);
                widen4<DT>(m[i].y, y0, y1);
                widen4<DT>(m[i].w, w0, w1);
                mma_dt<DT>(acc[i], y0, w0, y1, w1, b1);
            }
        };
        auto odd = [&](uint2 b) {                            // 16 columns after the 32s
            uint2 w[NG];
#pragma unroll
            for (int i = 0; i < NG; ++i) w[i] = lds64(at + i * gap + q32 * 512 + lane * 8);
#pragma unroll
            for (int i = 0; i < NG; ++i) {
                uint32_t x0, x1, y0, y1;
                widen4<DT>(w[i].x, x0, x1);
                widen4<DT>(w[i].y, y0, y1);
                mma_dt<DT>(acc[i], x0, y0, x1, y1, b);
            }
        };
        if constexpr (SMALL) {
            if (q32 > 0) chunk(0, sb.full[0], sb.full[1]);
            if (q32 > 1) chunk(1, sb.full[2], sb.full[3]);
            else if (q16 & 1) odd(q32 ? sb.full[2] : sb.full[0]);
        } else {
#pragma unroll 1
            for (int c = 0; c < q32; ++c) chunk(c, bfrag(frag, 2 * c, lane), bfrag(frag, 2 * c + 1, lane));
            if (q16 & 1) odd(bfrag(frag, 2 * q32, lane));
        }
    } else {
        auto step = [&](int c, uint2 b) {                    // 16 columns
            uint4 m[NG];
#pragma unroll
            for (int i = 0; i < NG; ++i) m[i] = lds128(a16 + i * gap + c * 512);
#pragma unroll
            for (int i = 0; i < NG; ++i) mma_dt<DT>(acc[i], m[i].x, m[i].z, m[i].y, m[i].w, b);
        };
        if constexpr (SMALL) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c < q16) step(c, sb.full[c]);
        } else {
#pragma unroll 2
            for (int c = 0; c < q16; ++c) step(c, bfrag(frag, c, lane));
        }
    }
    if (K & 15) {                                            // the last columns: 8, then pairs
        const uint2 b = SMALL ? sb.last : bfrag(frag, q16, lane);
        const int k8 = K & 8, pairs = (K & 7) >> 1;
        const uint32_t p8 = at + 16 * (K & ~15) * ES + lane * 4 * ES;
        const uint32_t pr = at + 16 * (K & ~7) * ES + ((lane >> 2) * pairs + (lane & 3)) * 4 * ES;
        const bool mine = (lane & 3) < pairs;
        uint2 u[NG], w[NG];
#pragma unroll
        for (int i = 0; i < NG; ++i) {
            u[i] = w[i] = make_uint2(0u, 0u);
            if (k8) {
                if constexpr (ES == 1) u[i].x = lds32(p8 + i * gap);
                else u[i] = lds64(p8 + i * gap);
            }
            if (mine) {
                if constexpr (ES == 1) w[i].x = lds32(pr + i * gap);
                else w[i] = lds64(pr + i * gap);
            }
        }
#pragma unroll
        for (int i = 0; i < NG; ++i) {
            if constexpr (ES == 1) {
                if (k8) widen4<DT>(u[i].x, u[i].x, u[i].y);
                widen4<DT>(w[i].x, w[i].x, w[i].y);
            }
            mma_dt<DT>(acc[i], u[i].x, u[i].y, w[i].x, w[i].y, b);
        }
    }
    // columns 0 and 1 of a row are on the quad's first lane, column 2 on its second
#pragma unroll
    for (int i = 0; i < NG; ++i)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float p2 = __shfl_xor_sync(0xffffffffu, acc[i][2 * r], 1);
            v[i][r] = HalfKind<DT>::v ? fmaf(fmaf(p2, 0x1p-11f, acc[i][2 * r + 1]), 0x1p-11f, acc[i][2 * r])
                                      : acc[i][2 * r] + (acc[i][2 * r + 1] + p2);
            // an infinite matrix entry (2-byte stores): the second and third parts may be zero, and
            // infinity times zero is no part of the sum
            if (ES == 2 && isinf(acc[i][2 * r])) v[i][r] = acc[i][2 * r];
        }
}

// The tiles of one slice in fragment order; returns the running tile count.  A warp
// takes the groups of 16 rows w, w + 14, ... of a tile, up to four at a time.  Each row's
// sum depends on the slice alone.  (The padding rows of the last group have their
// place in the partial vectors too: no row is tested.)  wide: set if the slice is marked
// (its sums come out as zeros and are replaced later).
template <int DT, bool SMALL>
__device__ __forceinline__ int consume_slice_frag(const Args& g, const Plan& pl, Shared& sh, int tid, int tile, int s,
                                                  int rb, int lo, bool& wide) {
    const int nact = g.nact, nst = g.nst, stage_bytes = g.stage_bytes;
    const int warp = tid >> 5, lane = tid & 31;
    const int K = rb / Esize<DT>::v;
    const float* frag = pl.bf + bfrag_floats(lo);
    SliceB sb{};
    if (SMALL) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (c < (K >> 4)) sb.full[c] = bfrag(frag, c, lane);
        if (K & 15) sb.last = bfrag(frag, K >> 4, lane);
    }
    const float down = pl.bscale[s - pl.sb0];
    wide |= down == 0.f;
    const bool first = (lane & 3) == 0;
    float* out = g.partial + static_cast<size_t>(s) * g.pstride + warp * 16 + (lane >> 2);
    const int tr = tile_rows(g, rb);
    const uint32_t gap = kConsumerWarps * 16 * rb, mine = pl.ring + warp * 16 * rb;
    int st = tile % nst, phase = (tile / nst) & 1;
    for (int row0 = 0; row0 < nact; row0 += tr, ++tile) {
        const bool ok = __all_sync(0xffffffffu, wait_phase(smem_addr(&sh.full_bar[st]), phase, &sh.abort_flag));
        if (ok) {
            const int ng = (min(tr, nact - row0) + 15) >> 4;
            uint32_t at = mine + st * stage_bytes;
            float* o = out + row0;
            auto take = [&](auto count) {                    // the warp's next groups
                constexpr int NG = decltype(count)::value;
                float v[NG][2];
                frag_dot<DT, NG, SMALL>(at, gap, K, lane, sb, frag, v);
                if (first)
#pragma unroll
                    for (int i = 0; i < NG; ++i)
#pragma unroll
                        for (int r = 0; r < 2; ++r)
                            o[i * kConsumerWarps * 16 + 8 * r] = HalfKind<DT>::v ? v[i][r] * down : v[i][r];
                at += NG * gap;
                o += NG * kConsumerWarps * 16;
            };
            int left = ng > warp ? (ng - warp + kConsumerWarps - 1) / kConsumerWarps : 0;
            for (; left >= 4; left -= 4) take(std::integral_constant<int, 4>());
            if (left & 2) take(std::integral_constant<int, 2>());
            if (left & 1) take(std::integral_constant<int, 1>());
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&sh.empty_bar[st]));
        } else if (lane == 0 && !sh.abort_flag) {
            // skip the work but keep reaching the block's barriers
            record_timeout(g);
            sh.abort_flag = 1;
        }
        if (++st == nst) {
            st = 0;
            phase ^= 1;
        }
    }
    return tile;
}

// A stored entry as FP32 (INT8 codes are stored flipped).
template <int DT>
__device__ __forceinline__ float stored_value(const unsigned char* p) {
    if constexpr (Esize<DT>::v == 2) {
        const unsigned short u = __ldg(reinterpret_cast<const unsigned short*>(p));
        return DT == RTC_BF16 ? __uint_as_float(static_cast<uint32_t>(u) << 16) : __half2float(__ushort_as_half(u));
    } else {
        const unsigned char u = __ldg(p);
        return DT == RTC_INT8 ? static_cast<float>(static_cast<int>(u) - 128) : e4m3x2_to_float2(u).x;
    }
}

// The rows of the block's marked slices as FP32 chains, from global memory: for a case too
// rare to hold registers or code in the loops above, and as near as the other sums.
template <int DT>
__device__ __forceinline__ void wide_slices(const Args& g, const Plan& pl, int tid) {
    constexpr int ES = Esize<DT>::v;
    consumer_sync();                                         // the sums that these replace are out
    for (int s = pl.sb0; s < pl.sb1; ++s) {
        if (pl.bscale[s - pl.sb0] != 0.f) continue;
        const int rb = __ldg(g.sl.rowbytes + s);
        const long long off = __ldg(g.sl.off + s);
        const float* sv = pl.loc + (__ldg(g.sl.loc + s) - pl.loc0);
        float* out = g.partial + static_cast<size_t>(s) * g.pstride;
        for (int row = tid; row < g.nact; row += kConsumers) {
            float acc = 0.f;
#pragma unroll 4
            for (int c = 0; c < rb / ES; ++c)
                acc = fmaf(stored_value<DT>(g.M + slice_elem_offset(off, rb, row, c * ES, ES)), sv[c], acc);
            out[row] = acc;
        }
    }
}

// One row of a fragment-order slice of K columns on the CUDA cores: row r of the group of
// 16 rows at shared address at, its terms added in column order.
template <int DT>
__device__ __forceinline__ float chain_row(uint32_t at, int K, int r, const float* sv) {
    constexpr int ES = Esize<DT>::v;
    const int g8 = r & 7, half = r >> 3;
    // <a 4-byte word, or its lower half, its slopes>; INT8 codes are stored flipped
    auto word = [](float acc, uint32_t w, const float* s) {
        return word_dot<DT>(acc, DT == RTC_INT8 ? w ^ 0x80808080u : w, s);
    };
    auto pair = [&](float acc, uint32_t a, const float* s) {
        if constexpr (ES == 2) return word(acc, lds32(a), s);
        else {
            const uint32_t w = lds16(a);
            const float2 p = DT == RTC_INT8 ? make_float2(i8_to_float(w, 0), i8_to_float(w, 1)) : e4m3x2_to_float2(w);
            return fmaf(p.y, s[1], fmaf(p.x, s[0], acc));
        }
    };
    float acc = 0.f;
    int c = 0;
    if constexpr (ES == 1)
        for (; c + 32 <= K; c += 32, at += 512)
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const uint2 w = lds64(at + ((g8 * 4 + t) * 2 + half) * 8);
                acc = word(word(acc, w.x, sv + c + 8 * t), w.y, sv + c + 8 * t + 4);
            }
    for (; c + 16 <= K; c += 16, at += 256 * ES)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const uint32_t a = at + ((g8 * 4 + t) * 2 + half) * 4 * ES;
            if constexpr (ES == 1) {
                acc = word(acc, lds32(a), sv + c + 4 * t);
            } else {
                const uint2 w = lds64(a);
                acc = word(word(acc, w.x, sv + c + 4 * t), w.y, sv + c + 4 * t + 2);
            }
        }
    if (c + 8 <= K) {
#pragma unroll
        for (int t = 0; t < 4; ++t) acc = pair(acc, at + ((g8 * 4 + t) * 2 + half) * 2 * ES, sv + c + 2 * t);
        at += 128 * ES;
        c += 8;
    }
    const int pairs = (K - c) >> 1;
    for (int t = 0; t < pairs; ++t) acc = pair(acc, at + ((g8 * pairs + t) * 2 + half) * 2 * ES, sv + c + 2 * t);
    return acc;
}

// The block's slices in fragment order by FP32 chains, a row a thread, each row's terms in
// column order; returns the running tile count.
template <int DT>
__device__ __forceinline__ int consume_chain(const Args& g, const Plan& pl, Shared& sh, int tid, int tile) {
    const int lane = tid & 31;
    for (int s = pl.sb0; s < pl.sb1; ++s) {
        const int rb = s == pl.sb0 ? pl.rb0 : __ldg(g.sl.rowbytes + s);
        const float* sv = pl.loc + (s == pl.sb0 ? 0 : __ldg(g.sl.loc + s) - pl.loc0);
        const int K = rb / Esize<DT>::v, tr = tile_rows(g, rb);
        float* out = g.partial + static_cast<size_t>(s) * g.pstride;
        for (int row0 = 0; row0 < g.nact; row0 += tr, ++tile) {
            const int st = tile % g.nst;
            if (__all_sync(0xffffffffu, wait_phase(smem_addr(&sh.full_bar[st]), (tile / g.nst) & 1, &sh.abort_flag))) {
                const uint32_t stage = pl.ring + st * g.stage_bytes;
                const int rows = min(tr, g.nact - row0);
                for (int r = tid; r < rows; r += kConsumers)
                    out[row0 + r] = chain_row<DT>(stage + (r >> 4) * 16 * rb, K, r & 15, sv);
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_addr(&sh.empty_bar[st]));
            } else if (lane == 0 && !sh.abort_flag) {
                record_timeout(g);
                sh.abort_flag = 1;
            }
        }
    }
    return tile;
}

// The consumer warps, after a consumer barrier that completes the block's slopes: every
// tile of the block's slices, one partial vector per
// slice (partial[s][row] = the row's dot product with the slice's slopes, in unit
// order).  tile0: the running tile count at entry; returns the count at exit.  The
// next slice's layout is fetched while the present one is consumed.  CHAIN: see
// chain_rule.
template <int DT, bool CHAIN>
__device__ __forceinline__ int consume(const Args& g, const Plan& pl, Shared& sh, int tid, int tile0) {
    if constexpr (CHAIN) return consume_chain<DT>(g, pl, sh, tid, tile0);
    int tile = tile0;
    int rb = pl.rb0, lo = 0;
    if constexpr (DT != RTC_F32) {
        make_bfrag<DT>(g, pl, tid);
        consumer_sync();
    }
    bool wide = false;                                       // the same on every thread
    for (int s = pl.sb0; s < pl.sb1; ++s) {
        int rb_next = 0, lo_next = 0;
        if (s + 1 < pl.sb1) {
            rb_next = __ldg(g.sl.rowbytes + s + 1);
            lo_next = __ldg(g.sl.loc + s + 1) - pl.loc0;
        }
        if constexpr (DT == RTC_F32) {
            const int u = row_unit(rb);
            if (u == 16) tile = consume_slice<DT, 16>(g, pl, sh, tid, tile, s, rb, lo);
            else if (u == 8) tile = consume_slice<DT, 8>(g, pl, sh, tid, tile, s, rb, lo);
            else tile = consume_slice<DT, 4>(g, pl, sh, tid, tile, s, rb, lo);
        } else {
            tile = rb <= 64 * Esize<DT>::v ? consume_slice_frag<DT, true>(g, pl, sh, tid, tile, s, rb, lo, wide)
                                           : consume_slice_frag<DT, false>(g, pl, sh, tid, tile, s, rb, lo, wide);
        }
        rb = rb_next;
        lo = lo_next;
    }
    if constexpr (DT != RTC_F32)
        if (wide) wide_slices<DT>(g, pl, tid);
    return tile;
}

// After the grid barrier that follows every block's partials: the rows [r0, r1) of
// the block, 32 at a time (one per lane), each summed over the S slices in a fixed
// order -- warp w adds the slices w, w+14, w+28, ... in turn (coalesced loads of 32
// consecutive rows of one slice), then warp 0 adds the 14 warp sums in a pairwise
// tree -- then the row scale and the integrator.  dm_out: where the new commands go
// besides g.a.
template <int DT>
__device__ __forceinline__ void reduce_rows(const Args& g, const Plan& pl, int tid,
                                            float* __restrict__ dm_out) {
    const int warp = tid >> 5, lane = tid & 31;
    for (int base = pl.r0; base < pl.r1; base += 32) {
        const int row = base + lane;
        float v = 0.f;
        if (row < pl.r1) {
            float p[kSlicesPerWarp];
#pragma unroll
            for (int j = 0; j < kSlicesPerWarp; ++j) {
                const int s = warp + j * kConsumerWarps;
                p[j] = s < g.sl.S ? __ldcg(g.partial + static_cast<size_t>(s) * g.pstride + row) : 0.f;
            }
#pragma unroll
            for (int j = 0; j < kSlicesPerWarp; ++j)
                if (warp + j * kConsumerWarps < g.sl.S) v += p[j];
        }
        pl.red[warp * 32 + lane] = v;
        consumer_sync();
        if (warp == 0 && row < pl.r1) {
            float t[kConsumerWarps];
#pragma unroll
            for (int w = 0; w < kConsumerWarps; ++w) t[w] = pl.red[w * 32 + lane];
#pragma unroll
            for (int width = 1; width < kConsumerWarps; width <<= 1)
#pragma unroll
                for (int i = 0; i + width < kConsumerWarps; i += 2 * width) t[i] += t[i + width];
            // the shared copy of the state stays current for a persistent kernel
            pl.a_pre[row - pl.r0] = integrate_row<DT>(row, t[0], pl.a_pre[row - pl.r0], pl.sc_pre[row - pl.r0],
                                                      g.a, dm_out, g.gain, g.leak);
        }
        consumer_sync();
    }
}

// What the sum over slices and the integrator of a per-frame call need.
struct SumArgs {
    const float* partial;    // [S][pitch]
    const float* scale;      // [nact] row scales, or null
    float* a;
    float* dm_out;           // [nact] or null
    int* status;             // for the caller's completion record
    int* cut;                // set if this step's partials are incomplete (record_timeout)
    unsigned* cutctr;        // finished blocks of a sum kernel that clears it (wraps)
    int S, nact, pitch;
    float gain, leak;
};

// Small systems: the whole sum by the last of the streaming blocks to finish, in its
// ring (drained by then), instead of by a kernel of its own.  No block waits for another.
// It takes 0.6 us longer on the GPU than the overlapped sum kernel at 4,000 values, but
// saves a launch, 1.4 us of the host's time, which is what bounds such frames.  Measured
// per frame in a stream of frames (two kernels -> this): 4,000 values (8x8) 9.0 -> 6.8 us,
// with prediction 10.9 -> 8.8; 7,000 (10x10) 8.9 -> 6.8; 15,000 (12x12) 8.9 -> 7.8, with
// prediction 10.9 -> 10.0; beyond that one block's loads take over: 34,000 (16x16) 8.8 ->
// 8.5 but 10.5 -> 11.3 with prediction, 58,000 (20x20) 8.9 -> 9.4.  A single frame from
// pinned host memory, whose launches overlap the GPU's work, does not gain (20.0 -> 20.1,
// 10x10 20.0 -> 20.5) and keeps the sum kernel.
constexpr int kLastSumValues = 16384;
constexpr int kLastSumGroups = 4;
constexpr size_t kLastSumSmem = 4 * static_cast<size_t>(kLastSumGroups) * kConsumerWarps * 32;
__host__ __device__ __forceinline__ bool last_block_sums(int S, int nact) { return S * nact <= kLastSumValues; }

// Called by every consumer once the block's partials are written; ctr counts the blocks
// of a launch and wraps.  The order of reduce_rows, four groups of 32 rows at a time.
__device__ __forceinline__ void last_block_sum(const SumArgs& r, unsigned* ctr, float* red, int* flag, int tid) {
    constexpr int kGroups = kLastSumGroups, kFlight = 11;
    const int warp = tid >> 5, lane = tid & 31;
    consumer_sync();
    if (tid == 0) {
        __threadfence();
        *flag = atomicInc(ctr, gridDim.x - 1) == gridDim.x - 1;
        __threadfence();
    }
    consumer_sync();
    if (!*flag) return;
    const bool ok = *reinterpret_cast<volatile int*>(r.cut) == RTC_OK;
    for (int base = 0; base < r.nact; base += 32 * kGroups) {
        const int row = base + 32 * warp + lane;             // of warps 0 .. kGroups - 1: their sums
        const bool mine = warp < kGroups && row < r.nact;
        const float a_prev = mine ? __ldcg(r.a + row) : 0.f;
        const float sc = mine && r.scale ? __ldg(r.scale + row) : 1.f;
        float v[kGroups] = {0.f, 0.f, 0.f, 0.f};
        for (int s0 = warp; s0 < r.S; s0 += kFlight * kConsumerWarps) {
            float p[kGroups][kFlight];
#pragma unroll
            for (int i = 0; i < kGroups; ++i)
#pragma unroll
                for (int j = 0; j < kFlight; ++j) {
                    const int s = s0 + j * kConsumerWarps, q = base + 32 * i + lane;
                    p[i][j] = s < r.S && q < r.nact ? __ldcg(r.partial + static_cast<size_t>(s) * r.pitch + q) : 0.f;
                }
#pragma unroll
            for (int i = 0; i < kGroups; ++i)
#pragma unroll
                for (int j = 0; j < kFlight; ++j)
                    if (s0 + j * kConsumerWarps < r.S) v[i] += p[i][j];
        }
#pragma unroll
        for (int i = 0; i < kGroups; ++i) red[(i * kConsumerWarps + warp) * 32 + lane] = v[i];
        consumer_sync();
        if (mine && ok) {
            float t[kConsumerWarps];
#pragma unroll
            for (int w = 0; w < kConsumerWarps; ++w) t[w] = red[(warp * kConsumerWarps + w) * 32 + lane];
#pragma unroll
            for (int width = 1; width < kConsumerWarps; width <<= 1)
#pragma unroll
                for (int i = 0; i + width < kConsumerWarps; i += 2 * width) t[i] += t[i + width];
            const float d = r.scale ? t[0] * sc : t[0];
            const float an = fmaf(r.leak, a_prev, r.gain * d);
            r.a[row] = an;
            if (r.dm_out) r.dm_out[row] = an;
        }
        consumer_sync();
    }
    if (tid == 0 && !ok) *r.cut = RTC_OK;        // every thread has read it
}

// Grid barrier over co-resident blocks: one thread per block, between two
// block-level barriers.  The arrival is a release and the polling an acquire at
// GPU scope, so the block's writes before the first block barrier are visible to
// every block after its second one (no separate fences).  The counter only grows;
// the caller passes the arrival count that completes this barrier.  False (and
// RTC_ETIMEDOUT in the status word) if it did not complete within kWaitNs.
//
// The two halves may also be called apart (grid_arrive, then grid_wait): loads the
// thread issues in between do not hold up its arrival, which a release would
// otherwise wait for.
__device__ __forceinline__ void grid_arrive(unsigned long long* bar) {
    asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(bar) : "memory");
}

__device__ __forceinline__ bool grid_wait(unsigned long long* bar, unsigned long long target, int* status,
                                          volatile int* abort) {
    const unsigned long long t0 = global_ns();
    while (true) {
        unsigned long long v;
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(bar) : "memory");
        if (v >= target) break;
        if (global_ns() - t0 > kWaitNs) {
            atomicExch(status, RTC_ETIMEDOUT);
            *abort = 1;
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ bool grid_barrier(unsigned long long* bar, unsigned long long target,
                                             int* status, volatile int* abort) {
    grid_arrive(bar);
    return grid_wait(bar, target, status, abort);
}

// One thread per block, after the block's commands are written: the last block to finish
// writes the completion record of a caller waiting on the host (every block, aborted or
// not, counts itself once).  A fence over the host link is a round trip, so there are two,
// the block's own and the record's release store (the other blocks' commands went out
// before they counted themselves; a fence on the device orders those counts): with two
// more, ELT frames from the host took 0.8 us longer, INT8 29.0 against 28.3.
__device__ __forceinline__ void finish_host(const FrameHost& fh, const int* status) {
    __threadfence_system();
    const unsigned long long prev = atomicAdd(fh.ctr, 1ull);
    if (prev + 1 == fh.target) {
        __threadfence();
        fh.done->status = *reinterpret_cast<const volatile int*>(status);
        asm volatile("st.release.sys.global.u64 [%0], %1;" ::"l"(&fh.done->seq), "l"(fh.seq) : "memory");
    }
}

// How much of the matrix a per-frame kernel requests when.  Its blocks start while the
// last frame's sum still has to read the partials and while their own pixels are not
// there; matrix traffic then delays both, but later there is too little time for it:
//   - the ring holds most of the block's share: nothing before the wait, since it fills
//     during the pixel stage anyway (ELT INT8 13.3 us against 13.9 with one tile early
//     and 14.1 with the whole ring; FP8 12.7, 13.2, 13.5);
//   - it holds less than half: one tile early, the rest of the ring at the wait and one
//     tile more into L2, which the HBM fetches during the pixel stage (ELT FP32 23.0 us
//     against 25.8 with the whole ring early and nothing ahead, BF16 16.5 against 17.4;
//     a lone frame with a cold L2 31.5 and 21.4 against 33.0 and 23.0.  Two tiles ahead
//     are 0.6 us better for BF16 frames one after another, but lone ones take 33.2 and
//     23.0);
//   - several pixel rounds a block (more sensors): the ring early and nothing ahead,
//     the pixel stage itself takes the HBM (six sensors FP8 47.8 us against 50).
//     Prediction frames too, whose blocks have the whole pixel kernel to wait for.
// (Against one cooperative kernel a frame every system between 8x8 and 74x74, with one to
// six sensors and every store, is faster under these rules, one frame after another and
// alone with cold caches.)
using Launch = LaunchPlan;

// Small slices of 1- and 2-byte stores: FP32 chains instead of the tensor cores.  Splitting
// the slopes, the two barriers around it and the fragments take 0.6 us whatever the size,
// and a thread's share of a small slice, its columns times the rows it takes, is less.
// Measured, loop (host to host) and frame after frame, INT8, tensor cores -> chains:
// 8x8 12.6 -> 11.4 and 6.5 -> 5.6 us, 26x26 (8 columns x 2 rows) 12.8 -> 12.4 and 6.1 ->
// 5.4, 34x34 (12 x 3) 13.1 -> 12.7 and 6.4 -> 6.0; beyond the line FP16 41x41 (18 x 4)
// 13.7 -> 14.0 and 6.9 -> 7.4, FP8 frames 6.8 -> 7.2.  INT8 converts more cheaply and has
// its line higher: 41x41 of 7 px 15.1 -> 14.7 and 7.0 -> 7.0.  Every slice of a matrix goes
// the same way, in all kernels.
constexpr int kChainSteps = 40, kChainStepsInt8 = 90;
template <int DT> struct CanChain { static constexpr bool v = DT != RTC_F32; };
inline bool chain_rule(int max_rb, int store, int esz, int nact) {
    const int steps = store == RTC_INT8 ? kChainStepsInt8 : kChainSteps;
    return esz < 4 && max_rb / esz * static_cast<long long>((nact + kConsumers - 1) / kConsumers) <= steps;
}
constexpr int kNoPredecessor = -1;

// min_region: shared-memory scratch a fused phase needs.  loop: the persistent kernel,
// which also sums its rows (integrator state, row scales and warp sums in shared
// memory); the lanes per row are the same for both.  Uses the handle's slice table,
// built when the matrix was loaded.
inline Launch plan_launch(const rtc_handle* h, size_t min_region = 0, bool loop = false) {
    Launch L{};
    const int S = h->sl_S;
    L.G = S < h->num_sms ? S : h->num_sms;
    if (L.G < 1 || S < 1 || static_cast<int>(h->sl_rowbytes.size()) != S) return L;
    // largest row and largest block-local slope vector over the blocks
    int max_rb = 0, max_loc = 0, max_floats = 0;
    const bool frag = h->sl_frag;
    const int esz = h->sl_esz;
    for (int b = 0; b < L.G; ++b) {
        const int s0 = static_cast<int>(static_cast<long long>(S) * b / L.G);
        const int s1 = static_cast<int>(static_cast<long long>(S) * (b + 1) / L.G);
        max_loc = std::max(max_loc, h->sl_loc[s1] - h->sl_loc[s0]);
        int floats = 0;
        for (int s = s0; s < s1; ++s) {
            max_rb = std::max(max_rb, h->sl_rowbytes[s]);
            floats += slope_floats(h->sl_g0[s + 1] - h->sl_g0[s], esz);
        }
        max_floats = std::max(max_floats, floats);
        L.max_slices = std::max(L.max_slices, s1 - s0);
    }
    L.loc_floats = (max_loc + 3) / 4 * 4;
    L.row_floats = (h->cfg.nact + L.G - 1) / L.G;
    L.region = (min_region + 15) / 16 * 16;
    L.chain = chain_rule(max_rb, h->store, esz, h->cfg.nact);
    L.bf_floats = frag ? bfrag_floats(L.loc_floats) : 0;
    const size_t slopes = 4 * static_cast<size_t>(L.loc_floats + L.bf_floats + (frag ? L.max_slices : 0));
    size_t extra = L.region + slopes + 8 * static_cast<size_t>(L.row_floats) + 4 * kConsumerWarps * 32;
    size_t budget = kDynSmemBudget;
    size_t room = budget > extra ? budget - extra : 0;
    // lanes per row: the fewest for which two stages of R = kConsumers / T rows fit
    // (splitting rows further to keep the slopes in registers measured slower for
    // every store type: more tiles and butterflies cost more than the slope reads
    // they save).  Only the slices decide it, not the block count, so the order of
    // every row's sum is the same for any launch of the handle.
    // In fragment order every row is one lane group's whatever the tile, so only the
    // tile shrinks (whole groups of 16 rows).
    auto rows_of = [&](int T) { return frag ? std::max(16, kConsumers / T / 16 * 16) : kConsumers / T; };
    auto stage = [&](int T) { return (static_cast<size_t>(rows_of(T)) * max_rb + 15) / 16 * 16; };
    L.T = 1;
    while (L.T < (frag ? 32 : 16) && 2 * stage(L.T) > room) L.T *= 2;      // R stays a multiple of 4
    L.R = rows_of(L.T);
    if (!loop) {
        extra = L.region + slopes;
        // (a plan that would not get its two stages beside a sum block takes the whole SM)
        budget = 2 * stage(L.T) + extra <= kFrameSmemBudget ? kFrameSmemBudget : kDynSmemBudget;
        room = budget > extra ? budget - extra : 0;
    }
    // stages of at least kMinTileBytes (whole multiples of R rows of the widest
    // slice), so that the per-tile handshakes stay a small part of the work
    const size_t st1 = stage(L.T);
    size_t m = st1 > 0 ? std::max<size_t>(1, (esz == 1 ? kMinTileBytes8 : kMinTileBytes) / st1) : 1;
    while (m > 1 && 2 * m * st1 > room) --m;
    L.stage_bytes = static_cast<int>(m * st1);
    const size_t fit = L.stage_bytes > 0 ? room / L.stage_bytes : 0;
    L.nst = static_cast<int>(fit < static_cast<size_t>(kMaxStages) ? fit : kMaxStages);
    L.smem = static_cast<size_t>(L.nst) * L.stage_bytes + extra;
    if (!loop && last_block_sums(S, h->cfg.nact)) L.smem = std::max(L.smem, kLastSumSmem);
    L.pre_tiles = loop ? kNoPredecessor : L.nst;
    if (!loop && min_region == 0 && h->n_valid * static_cast<long long>(h->cfg.n_wfs) <= 2ll * kConsumerWarps * L.G) {
        const bool most = 2ll * L.nst * L.stage_bytes * L.G >= h->m_bytes;
        L.pre_tiles = most ? 0 : 1;
        L.l2_ahead = most ? 0 : 1;
    }
    L.ok = L.nst >= 2 && max_floats <= kMaxLocalFloats && L.row_floats <= kMaxRowFloats &&
           S <= kMaxSlices && L.smem <= budget;
    if (frag) L.T = 1;
    return L;
}

// The plan of a per-frame kernel, worked out once per slice table and block limit: the
// walk over blocks and slices is 0.8 us of host time, a tenth of a small frame's call.
inline const Launch& frame_plan(rtc_handle* h, size_t pred_region, bool pred) {
    if (h->plan_sms != h->num_sms) {
        h->plan[0] = plan_launch(h);
        h->plan[1] = plan_launch(h, pred_region);
        h->plan_sms = h->num_sms;
    }
    return h->plan[pred ? 1 : 0];
}

inline Args make_args(const rtc_handle* h, const float* d_s, const Launch& L) {
    Args g{};
    g.M = static_cast<const unsigned char*>(h->d_M);
    g.sl = Slices{h->d_sl_off, h->d_sl_rowbytes, h->d_sl_g0, h->d_sl_loc, h->sl_S,
                  h->sl_S > 0 ? h->sl_g0[h->sl_S] : 0, h->sl_equal ? 1 : 0};
    g.nact = h->cfg.nact;
    g.n_valid = h->n_valid;
    g.T = L.T;
    g.R = L.R;
    g.stage_bytes = L.stage_bytes;
    g.nst = L.nst;
    g.l2_policy = h->m_bytes <= kL2KeepBytes ? kL2Normal : kL2Stream;
    g.region = static_cast<int>(L.region);
    g.frag = h->sl_frag ? 1 : 0;
    g.max_slices = L.max_slices;
    g.bf_floats = L.bf_floats;
    g.pre_tiles = L.pre_tiles;
    g.l2_ahead = L.l2_ahead;
    g.loc_floats = L.loc_floats;
    g.row_floats = L.row_floats;
    g.s = d_s;
    g.scale = h->d_scale;
    g.partial = h->d_partial;
    g.pstride = partial_pitch(h->cfg.nact);
    g.a = h->d_a;
    g.gain = h->gain;
    g.leak = h->leak;
    g.status = h->d_status;
    g.cut = h->d_status + 1;
    return g;
}

}  // namespace rtc_mvm

// Sum arguments of a handle (defined in mvm_stream.cu).
rtc_mvm::SumArgs sum_args(const rtc_handle* h, float* d_dm_out);
