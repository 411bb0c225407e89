// Back projection of libspect (sm_103a), FP32, first launch: the PSF and the
// attenuation of the transpose,
//   B_a[i][j][k] = A_a[i][j][k] * (K_i r_a)[j][k]   (K_i symmetric, zero padded)
// per angle, written to a rotated-frame volume that the adjoint-rotation
// gather (gather_tiled.cu, gather_kernel.cu) reads.
//
// One CTA per (depth chunk, z tile, angle, batch entry).  The projection r_a
// (with the tile's axial halo) is staged once; per depth plane the z-blur
// goes from it into a second buffer, and the j-blur strips are multiplied by
// A_i and stored.  Nothing of a plane's work is repeated for the halo, so the
// z tiles can be narrow and several CTAs share an SM.  Bound by FP32 FMA
// issue next to the HBM traffic of A and B; the rows of Q are a compile-time
// stride apart, so that the j-blur's loads need no address arithmetic.
#pragma once
#include "plane_common.cuh"

namespace spect {

namespace {

// zblur_strip with the taps loaded here.
template <int R>
__device__ __forceinline__ void zblur_row(const float4* out, const float* taps_row, float2 (&o)[kStrip])
{
    float2 w[R + 1];
    load_taps<R>(taps_row, w);
    zblur_strip<R>(out, w, o);
}

// A strip of kStrip rows of one column pair blurred along y into o (kFresh)
// or onto it: `out` is the column pair's quad in the strip's first row pair,
// row pairs kStride quads apart; the rows that the window reaches above and
// below the plane are zero rows of the buffer.
template <int R, bool kFresh, int kStride>
__device__ __forceinline__ void jblur_strip(const float4* out, const float* taps_row, float2 (&o)[kStrip])
{
    float2 w[R + 1];
    load_taps<R>(taps_row, w);
    const float4* src = out - window_lead<R>() * kStride;
    blur_pairs<R, kFresh>([&](int t) { return src[t * kStride]; }, o, w);
}

// z-blur of the staged projection P into Q, then the j-blur strips, each
// multiplied by A_i and stored.  A_i (the tile's columns, KT to a row) comes
// from the shared buffer (kSmemA: As, after waiting on `bar` with `parity`)
// or from global memory (aplane: row 0 of the tile's first column; nullptr
// without attenuation).  The radius R picks one of the unrolled strips.
// Returns false when the wait timed out.
template <int kSq, bool kSmemA, bool kHigh>
__device__ __forceinline__ bool back_blur_plane(int R, const float4* P, float4* Q, const BackTiling& t, int n, int nz,
                                                const ItemWalk& z_first, const ItemWalk& j_first,
                                                const float* taps_row, const float* As, uint32_t bar, uint32_t parity,
                                                const float* aplane, float* __restrict__ bplane, int KT)
{
    const int zstrips = t.ktpad / kStrip, jstrips = t.npad / kStrip;
#pragma unroll 1
    for (ItemWalk it = z_first; it.r < zstrips; it.next(t.zstep, t.npad >> 1)) {
        const float4* row = P + it.c * t.sp + (t.rh >> 1) + it.r * (kStrip / 2);
        float2 o[kStrip];
        switch (R) {
#define SPECT_BACK_CASE(RR) case RR: zblur_row<RR>(row, taps_row, o); break;
            SPECT_R_LOW(SPECT_BACK_CASE)
            default:
                if constexpr (kHigh) {
                    switch (R) {
                        SPECT_R_HIGH(SPECT_BACK_CASE)
                        default: break;
                    }
                }
#undef SPECT_BACK_CASE
        }
        store_zstrip(Q + it.c * kSq + it.r * (kStrip / 2), 1, o);
    }
    __syncthreads();
    // A_i was asked of L2 a plane ago and copied from there since the previous
    // plane ended; the z-blur covered it
    const bool ok = kSmemA ? mbar_wait(bar, parity) : true;
#pragma unroll 1
    for (ItemWalk it = j_first; it.r < jstrips; it.next(t.jstep, t.ktpad >> 1)) {
        const int kk = 2 * it.c, j0 = it.r * kStrip;
        const float4* out = Q + it.r * (kStrip / 2 * kSq) + it.c;
        float2 o[kStrip];
        switch (R) {
#define SPECT_BACK_CASE(RR) case RR: jblur_strip<RR, true, kSq>(out, taps_row, o); break;
            SPECT_R_LOW(SPECT_BACK_CASE)
            default:
                if constexpr (kHigh) {
                    switch (R) {
                        SPECT_R_HIGH(SPECT_BACK_CASE)
                        default: break;
                    }
                }
#undef SPECT_BACK_CASE
        }
        if (kk >= KT) continue;
        const size_t at = (size_t)j0 * nz + kk;
        float* bp = bplane + at;
        const float* ap = kSmemA ? As + j0 * KT + kk : aplane + at;
        const int astep = kSmemA ? KT : nz;
        if ((kSmemA || aplane) && j0 + kStrip <= n) {
            float2 av[kStrip];
#pragma unroll
            for (int r = 0; r < kStrip; ++r, ap += astep)
                av[r] = kSmemA ? *reinterpret_cast<const float2*>(ap) : __ldg(reinterpret_cast<const float2*>(ap));
#pragma unroll
            for (int r = 0; r < kStrip; ++r, bp += nz) *reinterpret_cast<float2*>(bp) = __fmul2_rn(o[r], av[r]);
        } else {
#pragma unroll
            for (int r = 0; r < kStrip; ++r, ap += astep, bp += nz) {
                if (j0 + r >= n) break;
                *reinterpret_cast<float2*>(bp) =
                    kSmemA || aplane ? __fmul2_rn(o[r], *reinterpret_cast<const float2*>(ap)) : o[r];
            }
        }
    }
    return ok;
}

}  // namespace

template <int kSq, bool kSmemA, bool kHigh>
__global__ void __launch_bounds__(kPlaneThreads, 1) blur_back_kernel(BlurBackArgs a)
{
    extern __shared__ __align__(16) float4 smem4[];
    const BackTiling& t = a.t;
    const int n = a.n, nz = a.nz;
    unsigned char* sm = reinterpret_cast<unsigned char*>(smem4);
    float4* P = smem4;
    float4* Q = reinterpret_cast<float4*>(sm + t.off_q) + t.pad_rows * kSq;  // row pairs from -pad_rows
    float* taps_s = reinterpret_cast<float*>(sm + t.off_taps);               // [2][kTapRow]
    float* As = reinterpret_cast<float*>(sm + t.off_a);
    const uint32_t bar = smem_u32(sm + t.off_bar);
    const int tid = threadIdx.x;
    const int chunk = blockIdx.x % a.chunks, tile = blockIdx.x / a.chunks;
    const int sidx = blockIdx.y, b = blockIdx.z;
    const int angle = a.sel[sidx];
    // this angle's PSF tables (a non-circular orbit has one per angle)
    const float* taps_g = a.taps + (size_t)angle * a.taps_stride;
    const int* rad_g = a.rad + (size_t)angle * a.rad_stride;
    const int* work_g = a.work + (size_t)angle * a.rad_stride;
    const int* bounds_g = a.bounds ? a.bounds + (size_t)angle * a.rad_stride : nullptr;
    const int kt0 = tile * t.ktile;
    const int KT = min(t.ktile, nz - kt0);
    const int kw0 = kt0 - t.rh;
    const int klo = max(0, kw0), khi = min(nz, kt0 + t.ktpad + t.rh);
    const size_t item = (size_t)b * a.n_sel + sidx;
    const float* aplane = a.atten ? a.atten + (size_t)angle * n * n * nz : nullptr;
    const int rp = t.npad >> 1;

    launch_dependents();

    // the j-blur's zero rows above and below the plane
    for (int it = tid; it < t.pad_rows * kSq; it += blockDim.x) {
        Q[it - t.pad_rows * kSq] = make_float4(0.f, 0.f, 0.f, 0.f);
        Q[it + rp * kSq] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    int i_lo, i_hi;
    chunk_planes(bounds_g, work_g, n, a.chunks, chunk, i_lo, i_hi);
    TapPrefetch tp;
    if (i_lo < i_hi) {
        tp.load(taps_g, i_lo);
        tp.store(taps_s, i_lo);
    }
    // a buffered plane is whole (one tile): one copy
    const uint32_t a_bytes = 4u * (uint32_t)(n * nz);
    if (kSmemA && tid == 0) {
        mbar_init(bar, 1);
        mbar_init_fence();
        if (i_lo < i_hi) tma_load_1d(smem_u32(As), aplane + (size_t)i_lo * n * nz, a_bytes, bar);
    }
    if (!kSmemA && aplane && i_lo < i_hi) prefetch_plane_l2(aplane + (size_t)i_lo * n * nz, n, nz, kt0, kt0 + KT);
    wait_prerequisites();  // up to here plan data only

    // The projection window of this angle (all ones without a projection),
    // times the angle's T_fov weights when the plan has them, zero outside
    // the detector.
    const float* pr = a.proj ? a.proj + (size_t)b * a.proj_bstride + (size_t)sidx * n * nz : nullptr;
    const float* fv = a.fov ? a.fov + (size_t)angle * n * nz : nullptr;
    const int wq = (t.ktpad >> 1) + t.rh;  // column pairs of the window
#pragma unroll 4
    for (int it = tid; it < rp * wq; it += blockDim.x) {
        const int jp = it / wq, cq = it - jp * wq;
        const int k = kw0 + 2 * cq;
        float2 v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = 2 * jp + h;
            v[h] = make_float2(0.f, 0.f);
            if (j < n && k >= klo && k < khi) {
                v[h] = pr ? *reinterpret_cast<const float2*>(pr + (size_t)j * nz + k) : make_float2(1.f, 1.f);
                if (fv) {
                    const float2 m = __ldg(reinterpret_cast<const float2*>(fv + (size_t)j * nz + k));
                    v[h] = make_float2(v[h].x * m.x, v[h].y * m.y);
                }
            }
        }
        P[jp * t.sp + cq] = make_float4(v[0].x, v[1].x, v[0].y, v[1].y);
    }
    __syncthreads();
    float* bvol = a.bvol + item * (size_t)n * n * nz;
    // this thread's first z-blur strip (row pair, strip) and j-blur strip
    // (column pair, strip)
    const ItemWalk z_first(rp), j_first(t.ktpad >> 1);
    uint32_t parity = 0;
    bool timed_out = false;
    int R = i_lo < i_hi ? __ldg(rad_g + i_lo) : 0;
    for (int i = i_lo; i < i_hi; ++i) {
        const int Rnext = i + 1 < i_hi ? __ldg(rad_g + i + 1) : 0;
        const size_t plane = (size_t)i * n * nz;
        if (i + 1 < i_hi) {
            tp.load(taps_g, i + 1);
            if (aplane) prefetch_plane_l2(aplane + plane + (size_t)n * nz, n, nz, kt0, kt0 + KT);
        }
        const bool ok = back_blur_plane<kSq, kSmemA, kHigh>(R, P, Q, t, n, nz, z_first, j_first,
                                                     taps_s + (i & 1) * kTapRow, As, bar, parity,
                                                     aplane ? aplane + plane + kt0 : nullptr, bvol + plane + kt0, KT);
        // the next plane's taps go to the half of taps_s read one plane ago
        if (i + 1 < i_hi) tp.store(taps_s, i + 1);
        R = Rnext;
        // Q is rewritten by the next plane's z-blur; A_i has been read
        if (!kSmemA) {
            __syncthreads();
            continue;
        }
        if (!sync_ok(ok, a.err)) {
            timed_out = true;
            break;
        }
        parity ^= 1;
        if (tid == 0 && i + 1 < i_hi) {
            fence_async_smem();
            tma_load_1d(smem_u32(As), aplane + plane + (size_t)n * nz, a_bytes, bar);
        }
    }
    // after a timed-out wait, give the copy in flight one more bounded wait
    // before the CTA (and its shared memory) goes away
    if (kSmemA && timed_out) mbar_wait(bar, parity);
}

namespace {
// Devices on which a kernel's shared-memory limit has been raised (at plan
// creation, so that launches inside a stream capture find it done).
template <int kSq, bool kSmemA, bool kHigh>
unsigned long long g_blur_back_smem_mask = 0;

template <int kSq, bool kSmemA, bool kHigh>
cudaError_t launch_sq(const BlurBackArgs& a, cudaStream_t st)
{
    cudaError_t e = allow_big_smem(blur_back_kernel<kSq, kSmemA, kHigh>, g_blur_back_smem_mask<kSq, kSmemA, kHigh>);
    if (e != cudaSuccess) return e;
    const dim3 grid(a.chunks * a.t.ntiles, a.n_sel, a.batch);
    return launch_early(blur_back_kernel<kSq, kSmemA, kHigh>, a, grid, a.t.threads, a.t.smem, st, 0, 1, a.early);
}

template <int kSq, bool kSmemA, bool kHigh>
int blocks_sq(const BackTiling& t)
{
    int blocks = 0;
    if (allow_big_smem(blur_back_kernel<kSq, kSmemA, kHigh>, g_blur_back_smem_mask<kSq, kSmemA, kHigh>) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, blur_back_kernel<kSq, kSmemA, kHigh>, t.threads, t.smem) !=
            cudaSuccess) {
        cudaGetLastError();  // do not leave the failure to a later launch check
        return 0;
    }
    return blocks;
}
}  // namespace

// One translation unit per (kSmemA, kHigh): blur_back_<v>.cu, in each one
// instantiation per row stride of kBackStrides.
#define SPECT_SQ_CASES(M)                                                                                     \
    case kBackStrides[0]: M(0); case kBackStrides[1]: M(1); case kBackStrides[2]: M(2);                       \
    case kBackStrides[3]: M(3); case kBackStrides[4]: M(4); case kBackStrides[5]: M(5);                       \
    case kBackStrides[6]: M(6)

template <bool kSmemA, bool kHigh>
cudaError_t launch_blur_back_v(const BlurBackArgs& a, cudaStream_t st)
{
    switch (a.t.sq) {
#define M(I) return launch_sq<kBackStrides[I], kSmemA, kHigh>(a, st)
        SPECT_SQ_CASES(M);
#undef M
        default: return cudaErrorInvalidValue;
    }
}

template <bool kSmemA, bool kHigh>
int blur_back_blocks_v(const BackTiling& t)
{
    switch (t.sq) {
#define M(I) return blocks_sq<kBackStrides[I], kSmemA, kHigh>(t)
        SPECT_SQ_CASES(M);
#undef M
        default: return 0;
    }
}

}  // namespace spect
