// Parts shared by the FP32 plane kernels (forward.cuh, blur_back.cuh): the
// separable PSF blur of one depth plane held in shared memory, its taps, and
// the split of the depth over CTAs.
//
// Packed arithmetic.  Both blur passes run on pairs of independent outputs
// with the sm_100-family paired FP32 FMA (__ffma2_rn: two IEEE fmaf in one
// instruction, so each result is bitwise a scalar fmaf): the z-blur on two
// rows (j, j+1) at once, the j-blur on two columns (k, k+1) at once.  The
// plane buffers therefore hold 2 x 2 quads (one float4 per row pair and
// column pair):
//   P  (z-blur input):  [row pair][column pair], quad
//      (P[j][k], P[j+1][k], P[j][k+1], P[j+1][k+1]), so one half of a quad
//      is the pair of rows at one column;
//   Q  (z-blurred plane, j-blur input): quad
//      (Z[j][k], Z[j][k+1], Z[j+1][k], Z[j+1][k+1]), so one half of a quad
//      is the pair of columns at one row; [column pair][row pair] in the
//      forward, [row pair][column pair] in the back blur.
// Lanes of a warp take consecutive row pairs (z-blur) or column pairs
// (j-blur), and the strides they step over are odd in 16-byte units, so the
// 128-bit shared-memory accesses of the blurs are free of bank conflicts.
#pragma once
#include <cuda_runtime.h>

#include "async_copy.cuh"
#include "geometry.cuh"
#include "internal.h"

namespace spect {

__device__ __forceinline__ float2 lo_half(const float4& q) { return make_float2(q.x, q.y); }
__device__ __forceinline__ float2 hi_half(const float4& q) { return make_float2(q.z, q.w); }

// kStrip output pairs of a 1-D blur:
//   o[q] += sum_m w(|q + R - m|) x[m],   m = 0 .. kStrip + 2R - 1,
// where input pair x[m] is half (m + (R & 1)) & 1 of the window's quad
// (m + (R & 1)) / 2 (the window starts one half early when R is odd).
// Sliding window: each loaded pair feeds up to 2R + 1 register accumulators.
// quad(t) returns the window's quad t.  kFresh: o starts at the first product
// instead of being added to.
template <int R, bool kFresh, class F>
__device__ __forceinline__ void blur_pairs(F&& quad, float2 (&o)[kStrip], const float2 (&w)[R + 1])
{
    constexpr int odd = R & 1;
    constexpr int nq = (kStrip + 2 * R + odd + 1) / 2;
#pragma unroll
    for (int qd = 0; qd < nq; ++qd) {
        const float4 v4 = quad(qd);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int m = 2 * qd + h - odd;
            if (m < 0 || m >= kStrip + 2 * R) continue;
            const float2 v = h ? hi_half(v4) : lo_half(v4);
#pragma unroll
            for (int q = 0; q < kStrip; ++q) {
                const int u = q + R - m;
                if (u < -R || u > R) continue;
                if (kFresh && u == R)  // the first input of output q
                    o[q] = __fmul2_rn(w[R], v);
                else
                    o[q] = __ffma2_rn(w[u < 0 ? -u : u], v, o[q]);
            }
        }
    }
}

// Quads between the start of a strip's window and its first output quad.
template <int R>
__host__ __device__ constexpr int window_lead()
{
    return (R + (R & 1)) / 2;
}

// Taps w(0..R) of a plane from its shared-memory row (see TapPrefetch),
// doubled in registers for the paired FMA.  (Rows that hold them doubled save
// the moves, but the wider loads cost registers: the blur then spills, and a
// spill is slow next to the little L1 that these kernels leave.)
template <int R>
__device__ __forceinline__ void load_taps(const float* row, float2 (&w)[R + 1])
{
#pragma unroll
    for (int q = 0; q <= R; ++q) {
        const float v = row[q];
        w[q] = make_float2(v, v);
    }
}

// The taps of the next plane travel through one register per thread (threads
// 0..kMaxR): loaded from global memory when a plane starts, stored to the
// other half of a two-row shared buffer when it ends, so that the load's
// latency hides behind the plane's work.  Rows hold w(0..kMaxR).
struct TapPrefetch {
    float v = 0.f;
    __device__ __forceinline__ void load(const float* __restrict__ taps, int plane)
    {
        if (threadIdx.x <= kMaxR) v = __ldg(taps + (size_t)plane * kTapW + kMaxR + threadIdx.x);
    }
    __device__ __forceinline__ void store(float* buf, int plane) const
    {
        if (threadIdx.x <= kMaxR) buf[(plane & 1) * kTapRow + threadIdx.x] = v;
    }
};

// Ask L2 to fetch columns [klo, khi) of every row of an attenuation plane
// ahead of its use, one 128-byte line per request (a hint per lane: the bulk
// form of the prefetch is issued lane by lane, a dozen instructions each).
// Rows and columns past the plane's end are not asked for.
__device__ __forceinline__ void prefetch_plane_l2(const float* plane, int n, int nz, int klo, int khi)
{
    if (klo == 0 && khi == nz) {  // the whole plane is one range
        const char* p = reinterpret_cast<const char*>(plane);
        const uint32_t bytes = (uint32_t)n * (uint32_t)nz * 4u;
        for (uint32_t o = 128u * threadIdx.x; o < bytes; o += 128u * blockDim.x) prefetch_line_l2(p + o);
        return;
    }
    for (int j = threadIdx.x; j < n; j += blockDim.x)
        for (int k = klo; k < khi; k += 32) prefetch_line_l2(plane + (size_t)j * nz + k);
}

// o = a strip of kStrip columns of one row pair blurred along z; `out`: the
// quad of the strip's first column in the row pair.
template <int R>
__device__ __forceinline__ void zblur_strip(const float4* out, const float2 (&w)[R + 1], float2 (&o)[kStrip])
{
    const float4* src = out - window_lead<R>();
    blur_pairs<R, true>([&](int t) { return src[t]; }, o, w);
}

// o[q] = (Z[j][k0+q], Z[j+1][k0+q]) as quads of a column pair and two rows,
// column pairs `step` quads apart.
__device__ __forceinline__ void store_zstrip(float4* dst, int step, const float2 (&o)[kStrip])
{
#pragma unroll
    for (int q = 0; q < kStrip; q += 2) dst[(q >> 1) * step] = make_float4(o[q].x, o[q + 1].x, o[q].y, o[q + 1].y);
}

// A thread's place in a grid of items, `width` to a row, that the CTA's
// threads walk in order: column `c` and row `r` of its current item, moved on
// without divisions (the steps are the launch's, ItemStep).
struct ItemWalk {
    int c, r;
    __device__ __forceinline__ explicit ItemWalk(int width) : c(threadIdx.x % width), r(threadIdx.x / width) {}
    __device__ __forceinline__ void next(const ItemStep& s, int width)
    {
        c += s.dc;
        r += s.dr;
        if (c >= width) {
            c -= width;
            ++r;
        }
    }
};

// Planes [lo, hi) of depth chunk `chunk`: the chunks split the prefix sums
// of the per-plane work estimate (staging plus both blur passes, which grow
// with 2R_i + 1) into equal parts.  A contiguous range keeps each CTA on one
// or two blur widths at a time, so an SM's instruction working set is one or
// two unrolled blur variants rather than all of them.  The prefix sums
// increase, so lo (hi) is the number of planes whose prefix lies below the
// chunk's start (end): counted by the whole CTA, one plane per thread.
// Every thread of the CTA must call this.
__device__ __forceinline__ void chunk_range(const int* __restrict__ work, int n, int chunks, int chunk, int& lo,
                                            int& hi)
{
    const long long total = __ldg(work + n);
    const long long start = total * chunk, end = total * (chunk + 1);
    lo = hi = 0;
    for (int i0 = 0; i0 < n; i0 += blockDim.x) {
        const int i = i0 + threadIdx.x;
        const long long v = i < n ? (long long)__ldg(work + i) * chunks : end;
        lo += __syncthreads_count(v < start);
        hi += __syncthreads_count(v < end);
    }
}

// The plane range of depth chunk `chunk`: from the host's boundary table
// (the contiguous split whose heaviest chunk is lightest) when it covers
// this chunk count, else chunk_range.  Every thread of the CTA must call it.
__device__ __forceinline__ void chunk_planes(const int* __restrict__ bounds, const int* __restrict__ work, int n,
                                             int chunks, int chunk, int& lo, int& hi)
{
    if (bounds && chunks <= kBoundChunks) {
        lo = __ldg(bounds + bound_offset(chunks) + chunk);
        hi = __ldg(bounds + bound_offset(chunks) + chunk + 1);
        return;
    }
    chunk_range(work, n, chunks, chunk, lo, hi);
}

// The radii the kernels unroll.  A plan whose radii are all at most kLowR
// takes kernels without the wider ones, whose taps cost every plane of a
// launch registers (and spills).
#define SPECT_R_LOW(M) M(0) M(1) M(2) M(3) M(4) M(5) M(6) M(7) M(8) M(9) M(10) M(11) M(12) M(13) M(14)
#define SPECT_R_HIGH(M) M(15) M(16) M(17) M(18) M(19) M(20)

// Raise the dynamic shared-memory limit of kernel `fn` to what the device
// allows next to the kernel's static shared memory, once per device.
template <class F>
inline cudaError_t allow_big_smem(F fn, unsigned long long& mask)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (mask & bit) return cudaSuccess;
    int optin = 0;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa{};
    e = cudaFuncGetAttributes(&fa, fn);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess) mask |= bit;
    return e;
}

}  // namespace spect
