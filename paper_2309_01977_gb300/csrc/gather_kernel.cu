// Transpose of the bilinear rotation (T_rot^T of Eq. 1) as a per-voxel
// gather, optionally fused with the OSEM update.
//
// For angle a and voxel column q = (x, y), the rotated-grid samples p whose
// bilinear footprint covers q lie in the box of half-width |cos|+|sin|
// around R(-theta)(q - c) + (c, cj) (cj: the angle's shifted detector centre).  The plan stores, per (angle, column), up to
// kMaxCand (offset of p's row in a rotated-frame volume, weight) pairs, the
// weight recomputed with the forward's own arithmetic so that it equals the
// forward weight bit for bit.  A convex region of area 4 and perimeter 8
// holds at most 4 + 8/2 + 1 = 9 lattice points, hence kMaxCand = 9.
#include <cuda_runtime.h>

#include "async_copy.cuh"
#include "geometry.cuh"
#include "internal.h"
#include "update.cuh"

namespace spect {

__global__ void gather_table_kernel(const float4* __restrict__ cs_tab, int n, int nz, int2* __restrict__ tab)
{
    const int angle = blockIdx.y;
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= n * n) return;
    const int x = col / n, y = col - x * n;
    const float c = 0.5f * (float)(n - 1);
    const float4 cs = cs_tab[angle];
    const float dx = (float)x - c, dy = (float)y - c;
    const float pi = c + cs.x * dx + cs.y * dy;
    const float pj = cs.z - cs.y * dx + cs.x * dy;
    const float ext = fabsf(cs.x) + fabsf(cs.y) + 1e-3f;
    const int ia = max(0, (int)ceilf(pi - ext)), ib = min(n - 1, (int)floorf(pi + ext));
    const int ja = max(0, (int)ceilf(pj - ext)), jb = min(n - 1, (int)floorf(pj + ext));
    int2* out = tab + ((size_t)angle * n * n + col) * kMaxCand;
    int count = 0;
    for (int i = ia; i <= ib; ++i)
        for (int j = ja; j <= jb; ++j) {
            float u, v;
            sample_point(cs.x, cs.y, c, cs.z, i, j, u, v);
            const float fu = floorf(u), fv = floorf(v);
            const int xa = (int)fu, ya = (int)fv;
            const float ax = u - fu, by = v - fv;
            const float wx = (x == xa) ? (1.f - ax) : (x == xa + 1 ? ax : 0.f);
            const float wy = (y == ya) ? (1.f - by) : (y == ya + 1 ? by : 0.f);
            if (wx != 0.f && wy != 0.f && count < kMaxCand) {
                out[count] = make_int2((i * n + j) * nz, __float_as_int(wx * wy));
                ++count;
            }
        }
    for (; count < kMaxCand; ++count) out[count] = make_int2(0, 0);
}

cudaError_t launch_gather_tables(const float4* cs, int n, int nz, int n_angles, int2* tab, cudaStream_t st)
{
    dim3 grid((n * n + 127) / 128, n_angles);
    gather_table_kernel<<<grid, 128, 0, st>>>(cs, n, nz, tab);
    return cudaGetLastError();
}

constexpr int kGatherThreads = 64;

// One warp per (voxel column, block of 32 float4 along z); with short columns
// (nz/4 < 32) a warp covers several columns, lanes_per_col lanes each.
// Angles are taken two at a time so that the table and volume loads of both
// are in flight together; the sum runs over angles in order, then over each
// angle's entries in table order, so it is deterministic.  Bound by the chain
// of loads: CTAs of two warps spread over the SMs in one wave.  kBlocks CTAs an
// SM cap the registers: 8 leave all loads of a pair of angles in flight at once,
// 16 twice the warps (see launch_gather).
template <int kBlocks>
__global__ void __launch_bounds__(kGatherThreads, kBlocks) gather_kernel(GatherArgs a)
{
    launch_dependents();
    const int n = a.n, nz = a.nz, zw = nz >> 2;
    const int lane = threadIdx.x & 31;
    const long gw = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    long col;
    int z4;
    if (a.lanes_per_col == 32) {
        const int zb = (zw + 31) >> 5;
        col = gw / zb;
        z4 = (int)(gw - col * zb) * 32 + lane;
    } else {
        col = gw * (32 / a.lanes_per_col) + lane / a.lanes_per_col;
        z4 = lane % a.lanes_per_col;
    }
    if (col >= (long)n * n || z4 >= zw) return;
    const int b = blockIdx.y;
    const size_t vol = (size_t)n * n * nz;
    const float* bb = a.bvol + (size_t)b * a.n_sel * vol + 4 * z4;
    const int2* __restrict__ tab = a.tab;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    // table entries of angle g (past the end: none)
    auto entries = [&](int g, int2 (&e)[kMaxCand]) {
        const bool in = g < a.n_sel;
        const int2* t = tab + ((size_t)a.sel[in ? g : 0] * n * n + col) * kMaxCand;
#pragma unroll
        for (int q = 0; q < kMaxCand; ++q) e[q] = in ? __ldg(t + q) : make_int2(0, 0);
    };
    wait_prerequisites();  // up to here plan data only
    for (int g = 0; g < a.n_sel; g += 2) {
        int2 e0[kMaxCand], e1[kMaxCand];
        entries(g, e0);
        entries(g + 1, e1);
        float4 v0[kMaxCand], v1[kMaxCand];
        float w0[kMaxCand], w1[kMaxCand];
        const float* b0 = bb + (size_t)g * vol;
        const float* b1 = bb + (size_t)(g + 1) * vol;
#pragma unroll
        for (int e = 0; e < kMaxCand; ++e) {
            w0[e] = __int_as_float(e0[e].y);
            w1[e] = __int_as_float(e1[e].y);
            v0[e] = e0[e].y != 0 ? *reinterpret_cast<const float4*>(b0 + e0[e].x) : make_float4(0.f, 0.f, 0.f, 0.f);
            v1[e] = e1[e].y != 0 ? *reinterpret_cast<const float4*>(b1 + e1[e].x) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        auto add = [&](float w, const float4& v) {
            if (w == 0.f) return;
            acc.x = fmaf(w, v.x, acc.x);
            acc.y = fmaf(w, v.y, acc.y);
            acc.z = fmaf(w, v.z, acc.z);
            acc.w = fmaf(w, v.w, acc.w);
        };
#pragma unroll
        for (int e = 0; e < kMaxCand; ++e) add(w0[e], v0[e]);
#pragma unroll
        for (int e = 0; e < kMaxCand; ++e) add(w1[e], v1[e]);
    }
    const bool upd = a.upd.mode != kUpdNone;
    const size_t i4 = ((size_t)col * nz >> 2) + z4;
    float4* o = reinterpret_cast<float4*>(a.out + (size_t)b * vol) + i4;
    float4 xv = make_float4(0.f, 0.f, 0.f, 0.f), sv = xv;
    if (upd || a.accumulate) xv = *o;
    if (upd) sv = reinterpret_cast<const float4*>(a.upd.sens)[i4];
    if (upd)
        *o = update4_sv(a.upd, xv, acc, sv, i4);
    else if (a.accumulate)
        *o = make_float4(xv.x + acc.x, xv.y + acc.y, xv.z + acc.z, xv.w + acc.w);
    else
        *o = acc;
}

cudaError_t launch_gather(const GatherArgs& a, cudaStream_t st)
{
    const int zw = a.nz >> 2;
    long warps;
    if (a.lanes_per_col == 32)
        warps = (long)a.n * a.n * ((zw + 31) / 32);
    else
        warps = ((long)a.n * a.n + (32 / a.lanes_per_col) - 1) / (32 / a.lanes_per_col);
    const long blocks = (warps * 32 + kGatherThreads - 1) / kGatherThreads;
    const dim3 grid((unsigned)blocks, a.batch);
    // 8 CTAs an SM where they hold a volume's warps in one wave, else 16.  12
    // angles in an OSEM run, us with the events around it, CTAs of 8 warps -> 8 CTAs
    // an SM / 16 (7 with the next pair's entries ahead): 40 x 36 16.0 -> 10.3 / 13.0
    // (12.3), 64^3 16.5 -> 13.0 / 14.5 (14.3), 57 x 80 17 -> 18.5 / 17.3 (18.5), 80
    // x 160 48 -> 53 / 45 (54), 112 x 136 90 -> 96 / 77 (102), 128 x 188 122 -> 131 /
    // 103 (136).
    if (warps <= 16L * a.num_sms) return launch_early(gather_kernel<8>, a, grid, kGatherThreads, 0, st);
    return launch_early(gather_kernel<16>, a, grid, kGatherThreads, 0, st);
}

}  // namespace spect
