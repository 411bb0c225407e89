// Forward projector of libspect (sm_103a), FP32.
//
// Eq. (1), one CTA per (depth chunk, z tile, angle, batch entry):
//   for each depth plane i of the chunk
//     stage   P[j][k] = A_a[i][j][k] * bilinear(f)(u(i,j), v(i,j), k)    (T_rot, T_att)
//     z-blur  Z[j][k] = sum_u w_i(u) P[j][k-u]                          (T_cdr, along z)
//     j-blur  acc[j][k] += sum_t w_i(t) Z[j-t][k]                       (T_cdr, along y; P_x)
//   The accumulator lives in registers for the whole depth loop.  With
//   several depth chunks per angle, each CTA stores a partial projection and
//   a separate reduction kernel adds the partials in chunk order (so the
//   result is deterministic) and, for OSEM, forms the ratio y / (p + s).
// The halo rh (the plan's largest PSF radius, rounded up to even) fixes the
// parity of a strip's window start, and so its quad boundaries, by R at
// compile time.
//
// Latency.  The attenuation plane of the next depth plane is copied into
// shared memory by a bulk copy (TMA, completing on an mbarrier) while the
// current plane is blurred, and the next plane's taps travel through one
// register; every wait is bounded and a timeout is reported in the plan's
// error word.
#pragma once
#include "plane_common.cuh"

namespace spect {

// z-blur item `it`: row pair jp, strip sidx of kStrip axial outputs.
// pq: quad offset in P of the item's first output position;
// qq: quad offset in Q of its first output (column pair 8*sidx, row pair jp).
struct ZItem {
    int pq, qq;
    bool valid;
};

__device__ __forceinline__ ZItem z_item(const PlaneTiling& t, int it)
{
    ZItem z;
    const int rp = t.npad >> 1;
    z.valid = it < rp * (t.ktpad / kStrip);
    const int jp = it % rp, sidx = it / rp;
    z.pq = jp * t.sp + ((t.rh + sidx * kStrip) >> 1);
    z.qq = sidx * (kStrip / 2) * t.sq + (t.rh >> 1) + jp;
    return z;
}

template <int R>
__device__ __forceinline__ void zblur_one(const float4* P, float4* Q, const PlaneTiling& t, const ZItem& z,
                                          const float2 (&w)[R + 1])
{
    float2 o[kStrip];
    zblur_strip<R>(P + z.pq, w, o);
    store_zstrip(Q + z.qq, t.sq, o);
}

// z-blur of the staged plane P into Q.  `z0` is this thread's first item;
// further items (more items than threads) are indexed here.
template <int R>
__device__ __forceinline__ void zblur_plane(const float4* P, float4* Q, const PlaneTiling& t, const ZItem& z0,
                                            const float2 (&w)[R + 1])
{
    if (z0.valid) zblur_one<R>(P, Q, t, z0, w);
    const int items = (t.npad >> 1) * (t.ktpad / kStrip);
    for (int it = threadIdx.x + blockDim.x; it < items; it += blockDim.x) zblur_one<R>(P, Q, t, z_item(t, it), w);
}

// j-blur item `it`: column pair kp = it % (ktpad/2), strip js of kStrip rows;
// the quad offset in Q of the strip's first output position, or -1.
__device__ __forceinline__ int j_item(const PlaneTiling& t, int it)
{
    const int cp = t.ktpad >> 1;
    if (it >= cp * (t.npad / kStrip)) return -1;
    const int kp = it % cp, js = it / cp;
    return kp * t.sq + ((t.rh + js * kStrip) >> 1);
}

template <int R, int IPT>
__device__ __forceinline__ void fwd_blur_plane(const float4* P, float4* Q, const PlaneTiling& t, const ZItem& z0,
                                               const int (&jq)[IPT], const float* taps_row,
                                               float2 (&acc)[IPT][kStrip])
{
    float2 w[R + 1];
    load_taps<R>(taps_row, w);
    zblur_plane<R>(P, Q, t, z0, w);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < IPT; ++q) {
        if (jq[q] < 0) continue;
        const float4* src = Q + jq[q] - window_lead<R>();
        blur_pairs<R, false>([&](int u) { return src[u]; }, acc[q], w);
    }
}

// Zero the column pairs of P outside the volume (the z-blur's zero padding)
// and, in every column pair of Q, the row-pair halo outside the rows the
// z-blur writes (the j-blur's zero padding).
__device__ __forceinline__ void zero_pads(float4* P, float4* Q, const PlaneTiling& t, int nz, int kw0)
{
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const int wq = (t.ktpad >> 1) + t.rh;  // column pairs of the window
    const int rp = t.npad >> 1, hq = t.rh >> 1;
    for (int idx = threadIdx.x; idx < rp * wq; idx += blockDim.x) {
        const int jp = idx / wq, cq = idx - jp * wq;
        const int k = kw0 + 2 * cq;
        if (k < 0 || k >= nz) P[jp * t.sp + cq] = z4;
    }
    const int qrows = rp + 2 * hq;
    for (int idx = threadIdx.x; idx < (t.ktpad >> 1) * qrows; idx += blockDim.x) {
        const int kp = idx / qrows, r = idx - kp * qrows;
        if (r < hq || r >= hq + rp) Q[kp * t.sq + r] = z4;
    }
}

// Bilinear taps of rotated row (i, j) of one plane, computed once per row
// by one thread and kept in shared memory: element offsets of the four tap
// rows in the volume and their weights.  Taps outside the grid get weight 0
// and offset 0, so every load stays in bounds.
struct TapRow {
    int off[4];
    float w[4];
};

__device__ __forceinline__ void tap_rows(TapRow* rows, int n, int nz, int i, float4 cs, float c)
{
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        float u, v;
        sample_point(cs.x, cs.y, c, cs.z, i, j, u, v);
        const float fu = floorf(u), fv = floorf(v);
        const int x0 = (int)fu, y0 = (int)fv;
        const float ax = u - fu, by = v - fv;
        const bool vx0 = x0 >= 0 && x0 < n, vx1 = x0 + 1 >= 0 && x0 + 1 < n;
        const bool vy0 = y0 >= 0 && y0 < n, vy1 = y0 + 1 >= 0 && y0 + 1 < n;
        TapRow t;
        t.w[0] = (vx0 && vy0) ? (1.f - ax) * (1.f - by) : 0.f;
        t.w[1] = (vx1 && vy0) ? ax * (1.f - by) : 0.f;
        t.w[2] = (vx0 && vy1) ? (1.f - ax) * by : 0.f;
        t.w[3] = (vx1 && vy1) ? ax * by : 0.f;
        t.off[0] = (vx0 && vy0) ? (x0 * n + y0) * nz : 0;
        t.off[1] = (vx1 && vy0) ? ((x0 + 1) * n + y0) * nz : 0;
        t.off[2] = (vx0 && vy1) ? (x0 * n + y0 + 1) * nz : 0;
        t.off[3] = (vx1 && vy1) ? ((x0 + 1) * n + y0 + 1) * nz : 0;
        rows[j] = t;
    }
}

// Sources of one rotated row (i, j) from column klo on: the four tap rows of
// the volume, their weights and the attenuation row (global memory, or the
// shared-memory copy of the plane).
struct RowSrc {
    const float* f[4];
    float w[4];
    const float* a;
};

__device__ __forceinline__ RowSrc row_src(const TapRow* rows, int j, const float* xb, const float* arow, int astride,
                                          int aoff, int klo)
{
    RowSrc r;
    const TapRow tr = rows[j];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        r.f[q] = xb + tr.off[q] + klo;
        r.w[q] = tr.w[q];
    }
    r.a = arow ? arow + (size_t)j * astride + aoff : nullptr;
    return r;
}

// The row's values at columns klo + c and klo + c + 1 (c even).  The first
// product is a plain multiply and the rest fmaf, in tap order, with the
// attenuation applied last, in the same order for every column.
template <bool kSmemA>
__device__ __forceinline__ float2 row_pair_value(const RowSrc& r, int c)
{
    const float2 f0 = *reinterpret_cast<const float2*>(r.f[0] + c);
    float2 v = __fmul2_rn(make_float2(r.w[0], r.w[0]), f0);
#pragma unroll
    for (int q = 1; q < 4; ++q) {
        const float2 f = *reinterpret_cast<const float2*>(r.f[q] + c);
        v = __ffma2_rn(make_float2(r.w[q], r.w[q]), f, v);
    }
    if (r.a) {
        const float2 a = kSmemA ? *reinterpret_cast<const float2*>(r.a + c)
                                : __ldg(reinterpret_cast<const float2*>(r.a + c));
        v = __fmul2_rn(v, a);
    }
    return v;
}

// The row's values at columns klo + c .. klo + c + 3 (c a multiple of 4;
// 16-byte aligned loads), each with the arithmetic of row_pair_value.
template <bool kSmemA>
__device__ __forceinline__ float4 row_quad_value(const RowSrc& r, int c)
{
    const float4 f0 = *reinterpret_cast<const float4*>(r.f[0] + c);
    const float2 w0 = make_float2(r.w[0], r.w[0]);
    float2 lo = __fmul2_rn(w0, make_float2(f0.x, f0.y)), hi = __fmul2_rn(w0, make_float2(f0.z, f0.w));
#pragma unroll
    for (int q = 1; q < 4; ++q) {
        const float4 f = *reinterpret_cast<const float4*>(r.f[q] + c);
        const float2 w = make_float2(r.w[q], r.w[q]);
        lo = __ffma2_rn(w, make_float2(f.x, f.y), lo);
        hi = __ffma2_rn(w, make_float2(f.z, f.w), hi);
    }
    if (r.a) {
        const float4 a = kSmemA ? *reinterpret_cast<const float4*>(r.a + c)
                                : __ldg(reinterpret_cast<const float4*>(r.a + c));
        lo = __fmul2_rn(lo, make_float2(a.x, a.y));
        hi = __fmul2_rn(hi, make_float2(a.z, a.w));
    }
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// P quads of every row pair over columns [klo, khi) (both even), from the
// row table: one row pair per warp at a time, lanes on consecutive column
// pairs.  Rows at or past n are zero.  In a partial last pass the column is
// clamped so that the loads stay in bounds; only the stores are masked.
// arow: attenuation of row 0 at column klo is arow[aoff], rows astride apart.
template <bool kSmemA>
__device__ __forceinline__ void stage_plane(float4* P, const PlaneTiling& t, const TapRow* rows,
                                            const float* __restrict__ xb, const float* arow, int astride, int aoff,
                                            int n, int kw0, int klo, int khi)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int ncols = khi - klo;
    // A row that fits one pass of 16-byte loads (4 columns per lane), with
    // every source row and the attenuation row 16-byte aligned at klo: half
    // the load instructions of the 8-byte path below, the same values.
    const bool wide = ncols <= 128 && (ncols & 3) == 0 && (klo & 3) == 0 && (aoff & 3) == 0 && (astride & 3) == 0;
    if (wide) {
        for (int jp = warp; jp < (t.npad >> 1); jp += nw) {
            float4* prow = P + jp * t.sp + ((klo - kw0) >> 1);
            const int j0 = 2 * jp, j1 = 2 * jp + 1;
            const int c4 = 4 * lane;
            if (j0 >= n) {
                if (c4 < ncols) {
                    prow[c4 >> 1] = make_float4(0.f, 0.f, 0.f, 0.f);
                    prow[(c4 >> 1) + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                continue;
            }
            const RowSrc r0 = row_src(rows, j0, xb, arow, astride, aoff, klo);
            const RowSrc r1 = row_src(rows, j1 < n ? j1 : j0, xb, arow, astride, aoff, klo);
            const int x4 = min(c4, ncols - 4);
            const float4 v0 = row_quad_value<kSmemA>(r0, x4);
            float4 v1 = row_quad_value<kSmemA>(r1, x4);
            if (j1 >= n) v1 = make_float4(0.f, 0.f, 0.f, 0.f);
            if (c4 < ncols) {
                prow[c4 >> 1] = make_float4(v0.x, v1.x, v0.y, v1.y);
                prow[(c4 >> 1) + 1] = make_float4(v0.z, v1.z, v0.w, v1.w);
            }
        }
        return;
    }
    for (int jp = warp; jp < (t.npad >> 1); jp += nw) {
        float4* prow = P + jp * t.sp + ((klo - kw0) >> 1);
        const int j0 = 2 * jp, j1 = 2 * jp + 1;
        if (j0 >= n) {
            for (int c = 2 * lane; c < ncols; c += 64) prow[c >> 1] = make_float4(0.f, 0.f, 0.f, 0.f);
            continue;
        }
        const RowSrc r0 = row_src(rows, j0, xb, arow, astride, aoff, klo);
        const RowSrc r1 = row_src(rows, j1 < n ? j1 : j0, xb, arow, astride, aoff, klo);
        // two 64-column passes at a time, so that all their loads are in
        // flight together
        for (int c0 = 0; c0 < ncols; c0 += 128) {
            const int ca = c0 + 2 * lane, cb = ca + 64;
            const int xa = min(ca, ncols - 2), xbb = min(cb, ncols - 2);
            const float2 a0 = row_pair_value<kSmemA>(r0, xa), b0 = row_pair_value<kSmemA>(r0, xbb);
            float2 a1 = row_pair_value<kSmemA>(r1, xa), b1 = row_pair_value<kSmemA>(r1, xbb);
            if (j1 >= n) a1 = b1 = make_float2(0.f, 0.f);
            if (ca < ncols) prow[ca >> 1] = make_float4(a0.x, a1.x, a0.y, a1.y);
            if (cb < ncols) prow[cb >> 1] = make_float4(b0.x, b1.x, b0.y, b1.y);
        }
    }
}

template <int IPT, bool kHigh>
__global__ void __launch_bounds__(kPlaneThreads, 1) forward_kernel(ForwardArgs a)
{
    extern __shared__ __align__(16) float4 smem4[];
    const PlaneTiling& t = a.t;
    const int n = a.n, nz = a.nz;
    unsigned char* sm = reinterpret_cast<unsigned char*>(smem4);
    float4* P = smem4;
    float4* Q = P + (size_t)(t.npad >> 1) * t.sp;
    TapRow* rows = reinterpret_cast<TapRow*>(Q + (size_t)(t.ktpad >> 1) * t.sq);
    float* taps_s = reinterpret_cast<float*>(sm + t.off_taps);  // [2][kTapRow]
    const int tid = threadIdx.x;
    const int chunk = blockIdx.x % a.chunks, tile = blockIdx.x / a.chunks;
    const int sidx = blockIdx.y, b = blockIdx.z;
    const int angle = a.sel[sidx];
    // this angle's PSF tables (a non-circular orbit has one per angle)
    const float* taps_g = a.taps + (size_t)angle * a.taps_stride;
    const int* rad_g = a.rad + (size_t)angle * a.rad_stride;
    const int* work_g = a.work + (size_t)angle * a.rad_stride;
    const int* bounds_g = a.bounds ? a.bounds + (size_t)angle * a.rad_stride : nullptr;
    const float4 cs = a.cs[angle];
    const float c = 0.5f * (float)(n - 1);
    const int kt0 = tile * t.ktile;
    const int KT = min(t.ktile, nz - kt0);
    const int kw0 = kt0 - t.rh;
    const int W = t.ktpad + 2 * t.rh;
    const int klo = max(0, kw0), khi = min(nz, kw0 + W);
    const float* aplane = a.atten ? a.atten + (size_t)angle * n * n * nz : nullptr;
    // attenuation planes through shared memory when the buffer fits
    const bool abuf = aplane && t.smem_a;
    const uint32_t a_bytes = 4u * (uint32_t)(n * nz);  // a buffered plane is whole (one tile)
    float* As = reinterpret_cast<float*>(sm + t.off_a);
    const uint32_t bar = smem_u32(sm + t.off_bar);
    launch_dependents();

    zero_pads(P, Q, t, nz, kw0);
    if (abuf && tid == 0) {
        mbar_init(bar, 1);
        mbar_init_fence();
    }

    // this thread's blur items, fixed for the whole depth loop
    const ZItem z0 = z_item(t, tid);
    int jq[IPT];
#pragma unroll
    for (int q = 0; q < IPT; ++q) jq[q] = j_item(t, tid + q * blockDim.x);

    float2 acc[IPT][kStrip];
#pragma unroll
    for (int q = 0; q < IPT; ++q)
#pragma unroll
        for (int r = 0; r < kStrip; ++r) acc[q][r] = make_float2(0.f, 0.f);

    const float* xb = a.x + (size_t)b * n * n * nz;
    int i_lo, i_hi;
    chunk_planes(bounds_g, work_g, n, a.chunks, chunk, i_lo, i_hi);
    TapPrefetch tp;
    if (i_lo < i_hi) {
        tp.load(taps_g, i_lo);
        tp.store(taps_s, i_lo);  // visible after the first barrier below
    }
    __syncthreads();  // barrier initialised
    if (abuf && tid == 0 && i_lo < i_hi)
        tma_load_1d(smem_u32(As), aplane + (size_t)i_lo * n * nz, a_bytes, bar);
    uint32_t parity = 0;
    bool timed_out = false;
    int R = i_lo < i_hi ? __ldg(rad_g + i_lo) : 0;
    wait_prerequisites();  // up to here plan data only
    for (int i = i_lo; i < i_hi; ++i) {
        const int Rnext = i + 1 < i_hi ? __ldg(rad_g + i + 1) : 0;  // a plane ahead
        if (i + 1 < i_hi) {
            tp.load(taps_g, i + 1);
            if (aplane && !abuf) prefetch_plane_l2(aplane + (size_t)(i + 1) * n * nz, n, nz, klo, khi);
        }
        // ---- stage the rotated, attenuated plane (T_rot, T_att)
        tap_rows(rows, n, nz, i, cs, c);
        bool ok = true;
        if (abuf) {
            ok = mbar_wait(bar, parity);  // A_i has landed
            parity ^= 1;
        }
        if (!sync_ok(ok, a.err)) {
            timed_out = true;
            break;
        }
        if (abuf)
            stage_plane<true>(P, t, rows, xb, As, nz, klo, n, kw0, klo, khi);
        else
            stage_plane<false>(P, t, rows, xb, aplane ? aplane + (size_t)i * n * nz : nullptr, nz, klo, n, kw0, klo,
                               khi);
        __syncthreads();
        // every read of A_i is done: fetch A_{i+1} behind the blur
        if (abuf && tid == 0 && i + 1 < i_hi) {
            fence_async_smem();
            tma_load_1d(smem_u32(As), aplane + (size_t)(i + 1) * n * nz, a_bytes, bar);
        }
        // ---- blur along z and y, accumulate over depth (T_cdr, P_x)
        const float* trow = taps_s + (i & 1) * kTapRow;
        switch (R) {
#define SPECT_FWD_CASE(RR) \
    case RR: fwd_blur_plane<RR, IPT>(P, Q, t, z0, jq, trow, acc); break;
            SPECT_R_LOW(SPECT_FWD_CASE)
            default:
                if constexpr (kHigh) {
                    switch (R) {
                        SPECT_R_HIGH(SPECT_FWD_CASE)
                        default: break;
                    }
                }
#undef SPECT_FWD_CASE
        }
        // The next plane's taps go to the other half of taps_s, last read
        // before this plane's second barrier.  The next staging writes P and
        // the row table only; Q is rewritten after the next two barriers,
        // which every thread reaches after its j-blur above.
        if (i + 1 < i_hi) tp.store(taps_s, i + 1);
        R = Rnext;
    }
    // after a timed-out wait, give the copy in flight one more bounded wait
    // before the CTA (and its shared memory) goes away
    if (timed_out) mbar_wait(bar, parity ^ 1);

    // Raw depth sums of this chunk: to the output when the chunk is the
    // whole depth and no ratio is wanted, else to the partial planes.
    const size_t item = (size_t)b * a.n_sel + sidx;
    float* dst = a.partials ? a.partials + (item * a.chunks + chunk) * (size_t)n * nz : a.out + item * (size_t)n * nz;
    const int cp = t.ktpad >> 1;
#pragma unroll
    for (int q = 0; q < IPT; ++q) {
        const int it = tid + q * blockDim.x;
        if (jq[q] >= 0) {
            const int kk = 2 * (it % cp), js = it / cp;
            if (kk < KT) {
#pragma unroll
                for (int r = 0; r < kStrip; ++r) {
                    const int j = js * kStrip + r;
                    if (j < n) *reinterpret_cast<float2*>(dst + (size_t)j * nz + kt0 + kk) = acc[q][r];
                }
            }
        }
    }
}

// ---------------------------------------------------------------- launchers

// Devices on which a kernel's shared-memory limit has been raised (shared by
// the occupancy query at plan creation and the launches, so that launches
// inside a stream capture find it done).
template <int IPT, bool kHigh>
unsigned long long g_forward_smem_mask = 0;
template <int IPT, bool kHigh>
cudaError_t forward_launch_ipt(const ForwardArgs& a, cudaStream_t st)
{
    cudaError_t e = allow_big_smem(forward_kernel<IPT, kHigh>, g_forward_smem_mask<IPT, kHigh>);
    if (e != cudaSuccess) return e;
    // The bilinear gathers live on L1: a launch of 32 angles at 192^3 takes 1.57 ms
    // with the smallest carve-out, 1.69 ms with the driver's choice; 160^3 x 8
    // 150 and 153 us.
    const dim3 grid(a.chunks * a.t.ntiles, a.n_sel, a.batch);
    return launch_early(forward_kernel<IPT, kHigh>, a, grid, a.t.threads, a.t.smem, st, a.t.ctas);
}

template <int IPT, bool kHigh>
int forward_occupancy_ipt(int threads, size_t smem)
{
    if (allow_big_smem(forward_kernel<IPT, kHigh>, g_forward_smem_mask<IPT, kHigh>) != cudaSuccess) {
        cudaGetLastError();  // do not leave the failure to a later launch check
        return 0;
    }
    int blocks = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, forward_kernel<IPT, kHigh>, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return blocks;
}

}  // namespace spect
