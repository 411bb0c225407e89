// Listmode PET system matrix H = T_eta T_omega P_Sigma T_rr (Sec. 2.1.1,
// Eq. (2)) and listmode OSEM (Table 1) on sm_103a.
//
// P_Sigma is Joseph's method: one thread per line of response walks the
// voxel planes of the line's principal axis and interpolates the image
// bilinearly in the other two axes.  The image (tens of MB) stays in L2
// across the walk, so the walk is bound by L2 request throughput, not HBM.
// Calls with enough lines therefore walk quads, the four taps of a sample as
// one 16-byte element (see pet_quad_kernel); the others walk the image.
// The listmode OSEM subiteration is a single pass over its events: each
// thread integrates its line through the blurred image, forms
// mult / (p + s) and spreads it back along the same samples with atomic adds
// (the expectation needs no other event, so no ratio array is written).
// T_rr is three separable 1-D passes; the last pass of the back projection
// applies the multiplicative update.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <map>
#include <string>
#include <vector>

#include "internal.h"
#include "pet.h"

namespace {

constexpr int kPetMaxR = 24;          // largest T_rr radius per axis
constexpr int kPetThreads = 256;
constexpr int kPetMaxBlocks = 152 * 32;

struct RrTaps {
    int r;                       // radius (0: identity)
    float w[2 * kPetMaxR + 1];   // w[t + r], t in [-r, r]
};

struct PetGrid {
    int n[3];
    float v[3];
    long long stride[3];  // elements between neighbours along x, y, z
    long long total;      // voxels
};

enum PetMode { kModeFwd = 0, kModeMult = 1, kModeBack = 2, kModeEm = 3 };

// The walk of one line: principal axis a, planes q0 .. q0 + count - 1, the
// in-plane index coordinates (u, w) on axes b < c at plane q0 and their
// increments per plane, and the step length (mm).
struct Walk {
    int a, b, c, q0, count;
    float u0, du, w0, dw, step;
    int i0, i1;       // samples visited (the time-of-flight window, else 0 .. count - 1)
    float l0, dl;     // arc length of sample 0 from the line's midpoint and its step (mm)
};

// Time of flight: bins of `width` mm centred at (b - (nb - 1)/2) width on the
// arc length from the line's midpoint (positive towards the second end);
// the Gaussian timing kernel integrated over the bin, truncated at
// nsigma sigma + width / 2.
struct TofParams {
    int nb;             // bins (0: no time of flight)
    float width, sigma, nsigma;
    float half_win;     // nsigma sigma + width / 2: the table covers [-half_win, half_win]
    float inv_h;        // table entries per mm
};

// The bin-integrated timing weight as a function of the distance x from the
// bin centre, tabulated at kTofTab + 1 points over [-half_win, half_win] and
// read with linear interpolation: the step is (2 nsigma + width / sigma)
// sigma / kTofTab, and the error (interpolation plus single-precision
// entries) stays near 4e-7 of the peak weight for bin widths of 0.5 to 2
// sigma.
constexpr int kTofTab = 4096;
constexpr size_t kTofSmem = (kTofTab + 1) * sizeof(float);

// Element i of a three-element array with constant indices only, so that
// the array stays in registers.
template <class T>
__device__ __forceinline__ T sel3(const T (&v)[3], int i)
{
    return i == 0 ? v[0] : i == 1 ? v[1] : v[2];
}

// The principal axis of a line, in single precision, rounded op by op.
__device__ __forceinline__ int line_axis(const float (&p1)[3], const float (&p2)[3], const PetGrid& g, float& scale)
{
    float sc[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) sc[c] = __fdiv_rn(fabsf(__fsub_rn(p2[c], p1[c])), g.v[c]);
    int a = 0;
    if (sc[1] > sc[0]) a = 1;
    if (sc[2] > sel3(sc, a)) a = 2;
    scale = sel3(sc, a);
    return a;
}

__device__ __forceinline__ void load_line(const float* __restrict__ lor, float (&p1)[3], float (&p2)[3])
{
    const float2 l0 = __ldg(reinterpret_cast<const float2*>(lor));
    const float2 l1 = __ldg(reinterpret_cast<const float2*>(lor) + 1);
    const float2 l2 = __ldg(reinterpret_cast<const float2*>(lor) + 2);
    p1[0] = l0.x;
    p1[1] = l0.y;
    p1[2] = l1.x;
    p2[0] = l1.y;
    p2[1] = l2.x;
    p2[2] = l2.y;
}

template <bool kTof>
__device__ __forceinline__ bool walk_setup(const float* __restrict__ lor, const PetGrid& g, Walk& k,
                                           const TofParams& tp, int bin, float& cb)
{
    float p1[3], p2[3];
    load_line(lor, p1, p2);
    // integer decisions in single precision
    float scale;
    const int a = line_axis(p1, p2, g, scale);
    if (!(scale > 0.f)) return false;
    const float va = sel3(g.v, a);
    const int na = sel3(g.n, a);
    const float half = __fmul_rn(0.5f, (float)(na - 1));
    const float org = -__fmul_rn(half, va);
    const float s1 = __fdiv_rn(__fsub_rn(sel3(p1, a), org), va);
    const float s2 = __fdiv_rn(__fsub_rn(sel3(p2, a), org), va);
    float lo = ceilf(s1 < s2 ? s1 : s2), hi = floorf(s1 < s2 ? s2 : s1);
    if (lo < 0.f) lo = 0.f;
    if (hi > (float)(na - 1)) hi = (float)(na - 1);
    if (!(lo <= hi)) return false;
    k.a = a;
    k.b = a == 0 ? 1 : 0;
    k.c = a == 2 ? 1 : 2;
    k.q0 = (int)lo;
    k.count = (int)hi - k.q0 + 1;
    // sample positions in double precision from the single-precision ends
    // (double operations spelled out where the time-of-flight window, an
    // integer, depends on their rounding)
    double e1[3], e2[3], len2 = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double v = (double)g.v[c];
        const double o = __dmul_rn(-0.5 * (double)(g.n[c] - 1), v);
        e1[c] = __ddiv_rn(__dsub_rn((double)p1[c], o), v);
        e2[c] = __ddiv_rn(__dsub_rn((double)p2[c], o), v);
        const double d = __dsub_rn((double)p2[c], (double)p1[c]);
        len2 = __dadd_rn(len2, __dmul_rn(d, d));
    }
    const double da = __dsub_rn(sel3(e2, a), sel3(e1, a));
    const double t0 = __ddiv_rn(__dsub_rn((double)k.q0, sel3(e1, a)), da);
    const double db = sel3(e2, k.b) - sel3(e1, k.b), dc = sel3(e2, k.c) - sel3(e1, k.c);
    k.u0 = (float)(sel3(e1, k.b) + t0 * db);
    k.w0 = (float)(sel3(e1, k.c) + t0 * dc);
    k.du = (float)(db / da);
    k.dw = (float)(dc / da);
    const double len = __dsqrt_rn(len2);
    k.step = (float)((double)va * len / fabs((double)sel3(p2, a) - (double)sel3(p1, a)));
    k.i0 = 0;
    k.i1 = k.count - 1;
    if (kTof) {
        const double l0 = __dmul_rn(__dsub_rn(t0, 0.5), len);
        const double dl = __ddiv_rn(len, da);
        const double width = (double)tp.width;
        const double c = __dmul_rn(__dsub_rn((double)bin, __dmul_rn(0.5, (double)(tp.nb - 1))), width);
        const double w = __dadd_rn(__dmul_rn((double)tp.nsigma, (double)tp.sigma), __dmul_rn(0.5, width));
        double lo = __ddiv_rn(__dsub_rn(__dsub_rn(c, w), l0), dl);
        double hi = __ddiv_rn(__dsub_rn(__dadd_rn(c, w), l0), dl);
        if (dl < 0.0) {
            const double t = lo;
            lo = hi;
            hi = t;
        }
        lo = ceil(lo);
        hi = floor(hi);
        if (lo < 0.0) lo = 0.0;
        if (lo > (double)k.count) lo = (double)k.count;
        if (hi > (double)(k.count - 1)) hi = (double)(k.count - 1);
        if (hi < -1.0) hi = -1.0;
        k.i0 = (int)lo;
        k.i1 = (int)hi;
        k.l0 = (float)l0;
        k.dl = (float)dl;
        cb = (float)c;
    }
    return true;
}

// The timing weight of sample i.
__device__ __forceinline__ float tof_weight(float l0, float dl, const TofParams& tp, float cb, const float* tof_tab,
                                            int i)
{
    const float x = (fmaf((float)i, dl, l0) - cb + tp.half_win) * tp.inv_h;
    const float xc = fminf(fmaxf(x, 0.f), (float)kTofTab);
    const int j = min((int)xc, kTofTab - 1);
    const float fr = xc - (float)j;
    const float t0 = tof_tab[j], t1 = tof_tab[j + 1];
    return fmaf(fr, t1 - t0, t0);
}

// Visits the in-image bilinear taps of every step-th sample from `first` on, one
// image row of the b axis at a time: fn(idx, ok0, ok1, w0, w1) for the taps idx (along c at
// iw) and idx + stride_c (at iw + 1), each present only where ok.
template <bool kTof, class F>
__device__ __forceinline__ void walk(const Walk& k, const PetGrid& g, const TofParams& tp, float cb,
                                     const float* tof_tab, int first, int step, F&& fn)
{
    const long long sa = sel3(g.stride, k.a), sb = sel3(g.stride, k.b), sc = sel3(g.stride, k.c);
    const int nb = sel3(g.n, k.b), nc = sel3(g.n, k.c);
    for (int i = first; i <= k.i1; i += step) {
        const float wt = kTof ? tof_weight(k.l0, k.dl, tp, cb, tof_tab, i) : 1.f;
        const float u = fmaf((float)i, k.du, k.u0);
        const float w = fmaf((float)i, k.dw, k.w0);
        const float fu = floorf(u), fw = floorf(w);
        // outside the image by a full voxel: no tap reads anything
        if (!(fu >= -1.f && fu <= (float)(nb - 1) && fw >= -1.f && fw <= (float)(nc - 1))) continue;
        const int iu = (int)fu, iw = (int)fw;
        const float tu = u - fu, tw = w - fw;
        const long long base = (long long)(k.q0 + i) * sa + (long long)iu * sb + (long long)iw * sc;
        const bool w0ok = iw >= 0, w1ok = iw + 1 < nc;
        const float ru = (1.f - tu) * wt, su = tu * wt;
        if (iu >= 0) fn(base, w0ok, w1ok, ru * (1.f - tw), ru * tw);
        if (iu + 1 < nb) fn(base + sb, w0ok, w1ok, su * (1.f - tw), su * tw);
    }
}

// w0 img[idx] + w1 img[idx + sc] over the present taps.  Two taps next to
// each other in memory (sc == 1) inside one aligned 16-byte quad of the
// image are read with one vector load.
__device__ __forceinline__ float gather_pair(const float* __restrict__ img, long long idx, long long sc,
                                             long long total, bool ok0, bool ok1, float w0, float w1)
{
    const long long q = idx & ~3LL;
    const int r = (int)(idx & 3);
    if (sc == 1 && ok0 && ok1 && r < 3 && q + 3 < total) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(img + q));
        const float a = r == 0 ? v.x : r == 1 ? v.y : v.z;
        const float b = r == 0 ? v.y : r == 1 ? v.z : v.w;
        return fmaf(w1, b, w0 * a);
    }
    float acc = 0.f;
    if (ok0) acc = w0 * __ldg(img + idx);
    if (ok1) acc = fmaf(w1, __ldg(img + idx + sc), acc);
    return acc;
}

// bp[idx] += v0, bp[idx + sc] += v1 over the present taps: one 16-byte
// vector atomic when both fall in one aligned quad (the other two lanes add
// +0, which leaves every non-negative value unchanged), else scalar atomics.
__device__ __forceinline__ void scatter_pair(float* bp, long long idx, long long sc, long long total, bool ok0,
                                             bool ok1, float v0, float v1)
{
    const long long q = idx & ~3LL;
    const int r = (int)(idx & 3);
    if (sc == 1 && ok0 && ok1 && r < 3 && q + 3 < total) {
        const float4 v = make_float4(r == 0 ? v0 : 0.f, r == 0 ? v1 : r == 1 ? v0 : 0.f,
                                     r == 1 ? v1 : r == 2 ? v0 : 0.f, r == 2 ? v1 : 0.f);
        atomicAdd(reinterpret_cast<float4*>(bp + q), v);
        return;
    }
    if (ok0) atomicAdd(bp + idx, v0);
    if (ok1) atomicAdd(bp + idx + sc, v1);
}

struct LmArgs {
    const float* img;     // image read by the walk (blurred x, or mu)
    float* bp;            // back-projection accumulator
    const float* lors;    // [n][6]
    const float* mult;    // [n] or nullptr (1)
    const float* vals;    // kModeBack: q [n]; kModeMult: eta [n] or nullptr
    const float* s;       // kModeEm: [n] or nullptr (0)
    float* out;           // kModeFwd / kModeMult: [n]
    double* diag;         // kModeEm: 2 doubles (sum p/(p+s), events used) or nullptr
    const int* tof_bin;   // [n] time-of-flight bins (kTof kernels)
    const float* tof_tab; // [kTofTab + 1] timing weights (kTof kernels)
    float4* quads;        // pet_quad_kernel: the image's quads of this axis (kModeBack: unused)
    float4* bquads;       // and the back projection's
    long long first, stride, count;  // events first + t * stride, t < count
    PetGrid g;
    TofParams tof;
};

__device__ __forceinline__ void block_add2(double a, double b, double* dst)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    __shared__ double red[2][kPetThreads / 32];  // the most warps of a block
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        red[0][wid] = a;
        red[1][wid] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double sa = 0.0, sb = 0.0;
        for (int i = 0; i < (int)blockDim.x / 32; ++i) {
            sa += red[0][i];
            sb += red[1][i];
        }
        atomicAdd(dst, sa);
        atomicAdd(dst + 1, sb);
    }
}

template <int kMode, bool kTof>
__global__ void __launch_bounds__(kPetThreads) pet_lm_kernel(LmArgs a)
{
    extern __shared__ float tof_s[];  // kTof: the timing-weight table
    if (kTof) {
        for (int i = threadIdx.x; i <= kTofTab; i += blockDim.x) tof_s[i] = __ldg(a.tof_tab + i);
        __syncthreads();
    }
    double cons = 0.0, used = 0.0;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < a.count;
         t += (long long)gridDim.x * blockDim.x) {
        const long long e = a.first + t * a.stride;
        Walk k;
        float cb = 0.f;
        const bool hit = walk_setup<kTof>(a.lors + 6 * e, a.g, k, a.tof, kTof ? __ldg(a.tof_bin + e) : 0, cb);
        if (kMode == kModeBack) {
            const float val = __ldg(a.vals + e) * (a.mult ? __ldg(a.mult + e) : 1.f);
            if (!hit || val == 0.f) continue;
            const float sv = val * k.step;
            const long long sc = sel3(a.g.stride, k.c);
            walk<kTof>(k, a.g, a.tof, cb, tof_s, k.i0, 1, [&](long long idx, bool o0, bool o1, float w0, float w1) {
                scatter_pair(a.bp, idx, sc, a.g.total, o0, o1, sv * w0, sv * w1);
            });
            continue;
        }
        float acc = 0.f;
        if (hit && (kMode != kModeMult || a.img != nullptr)) {
            const long long sc = sel3(a.g.stride, k.c);
            walk<kTof>(k, a.g, a.tof, cb, tof_s, k.i0, 1, [&](long long idx, bool o0, bool o1, float w0, float w1) {
                acc += gather_pair(a.img, idx, sc, a.g.total, o0, o1, w0, w1);
            });
        }
        const float line = hit ? acc * k.step : 0.f;
        if (kMode == kModeFwd) {
            a.out[e] = a.mult ? __ldg(a.mult + e) * line : line;
        } else if (kMode == kModeMult) {
            const float om = a.img ? expf(-line) : 1.f;
            a.out[e] = (a.vals ? __ldg(a.vals + e) : 1.f) * om;
        } else {  // kModeEm
            const float m = __ldg(a.mult + e);
            const float p = m * line;
            const float den = p + (a.s ? __ldg(a.s + e) : 0.f);
            if (!(den > 0.f)) continue;
            cons += (double)p / (double)den;
            used += 1.0;
            const float sv = m / den * k.step;
            if (hit) {
                const long long sc = sel3(a.g.stride, k.c);
                walk<kTof>(k, a.g, a.tof, cb, tof_s, k.i0, 1, [&](long long idx, bool o0, bool o1, float w0, float w1) {
                    scatter_pair(a.bp, idx, sc, a.g.total, o0, o1, sv * w0, sv * w1);
                });
            }
        }
    }
    if (kMode == kModeEm && a.diag) block_add2(cons, used, a.diag);
}

// ---------------------------------------------------------------- quads
//
// The plain walk costs 2.5 L2 requests a sample each way (a row's z-pair is
// one 16-byte access three times in four, else two), and the L2 serves them
// at its limit.  The quads of axis AX (0: x, 1: y; b the other of the two)
// hold for every plane q and every cell (iu, iw) of the (b, z) lattice, one
// cell past the image on each side, the four values f(iu, iw), f(iu, iw + 1),
// f(iu + 1, iw), f(iu + 1, iw + 1), zero outside the image: a sample's gather
// is one aligned 16-byte load without edge cases, its scatter one 16-byte
// vector atomic into an accumulator of the same shape, which a fold adds up
// per voxel afterwards.  The lines of one axis go together (x, then y), so
// that one axis's quads are in use at a time; lines along z, which a
// cylindrical scanner hardly has, walk the image.
// With a line of response to a lane and cells in plane order the walk was bound
// by L1's rate of one line a cycle: a warp's 32 lanes touched 32 lines a sample
// each way (1.7 cycles a sample for the gather, 2.0 for the scatter).  Four lanes
// now walk a line together, on consecutive planes, and the cells lie in
// 128-byte bricks of 4 planes x 2 u x 1 w, so that the four share about two
// lines (along the axis a line moves by half a cell in u and less in w).  What
// bounds it now is the latency of misses past L2: at 204 x 204 x 154 the two sets
// of quads are 104 MB each, 43 % of the sectors hit, and HBM moves 3.6 TB/s; L1
// and the issue slots are half busy.
// Measured, image walk -> quads in plane order -> bricks: an iteration of 3 M
// events in 3 subsets at 204 x 204 x 154 with time of flight 9.7 -> 6.95 ->
// 5.58 ms; 128 x 128 x 90, 1 M lines without, forward and back 2.60 -> 1.46 ->
// 1.23 ms.  64 registers (32 warps an SM at most, 28 on average) are worth more
// than a wider batch: 2.79 -> 2.20 ms a subset.  Tried and not better: gathering
// and scattering in separate launches (2.71 ms), the time-of-flight lines slab by
// slab along the axis (2.27 ms).

constexpr int kQuadThreads = 128;

// Where cell (u, w) of plane q lies in axis AX's lattice of na planes of
// (nb + 1) x (nz + 1) cells: bricks of 4 planes x 2 u, 128 bytes, side by side
// along w, the planes of one u next to each other in a brick.
struct QuadLattice {
    int w, u2, na4;  // cells along w, bricks along u and along the axis
};

__host__ __device__ inline QuadLattice quad_lattice(const PetGrid& g, int ax)
{
    return {g.n[2] + 1, (g.n[1 - ax] + 2) >> 1, (g.n[ax] + 3) >> 2};
}

__device__ __forceinline__ int quad_at(const QuadLattice& l, int q, int u, int w)
{
    return ((((q >> 2) * l.u2 + (u >> 1)) * l.w + w) << 3) + ((u & 1) << 2) + (q & 3);
}

__host__ __device__ inline long long quad_cells(const PetGrid& g, int ax)
{
    const QuadLattice l = quad_lattice(g, ax);
    return 8ll * l.na4 * l.u2 * l.w;
}

template <int AX>
__global__ void __launch_bounds__(kPetThreads) pet_quads_kernel(const float* __restrict__ img, float4* __restrict__ quads,
                                                                PetGrid g)
{
    const int na = g.n[AX], nb = g.n[1 - AX], nc = g.n[2];
    const int sb = AX == 0 ? nc : g.n[1] * nc, sa = AX == 0 ? g.n[1] * nc : nc;  // voxels < 2^31 (use_quads)
    const QuadLattice l = quad_lattice(g, AX);
    const int total = (int)quad_cells(g, AX);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < total; c += gridDim.x * blockDim.x) {
        const int k = c >> 3, w = k % l.w, r = k / l.w;
        const int u = (r % l.u2) * 2 + ((c >> 2) & 1), q = (r / l.u2) * 4 + (c & 3);
        if (q >= na || u > nb) continue;  // a brick's cells past the lattice: never read
        const float* p = img + (long long)q * sa + (long long)(u - 1) * sb + (w - 1);
        const bool u0 = u > 0, u1 = u < nb, w0 = w > 0, w1 = w < nc;
        quads[c] = make_float4(u0 && w0 ? __ldg(p) : 0.f, u0 && w1 ? __ldg(p + 1) : 0.f, u1 && w0 ? __ldg(p + sb) : 0.f,
                               u1 && w1 ? __ldg(p + sb + 1) : 0.f);
    }
}

// bp += the accumulated quads of axis AX.  Threads walk voxels in the order of
// the bricks (4 planes x 2 along b, then z), so that a warp's reads share lines.
template <int AX>
__global__ void __launch_bounds__(kPetThreads) pet_fold_kernel(const float4* __restrict__ quads, float* __restrict__ bp,
                                                               PetGrid g)
{
    const int na = g.n[AX], nb = g.n[1 - AX], nc = g.n[2];
    const int sb = AX == 0 ? nc : g.n[1] * nc, sa = AX == 0 ? g.n[1] * nc : nc;
    const QuadLattice l = quad_lattice(g, AX);
    const int b2 = (nb + 1) >> 1, total = 8 * l.na4 * b2 * nc;  // at most quad_cells
    const float* q1 = reinterpret_cast<const float*>(quads);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < total; c += gridDim.x * blockDim.x) {
        const int k = c >> 3, z = k % nc, r = k / nc;
        const int b = (r % b2) * 2 + ((c >> 2) & 1), q = (r / b2) * 4 + (c & 3);
        if (q >= na || b >= nb) continue;
        // cell (u, w) of the lattice is lattice point (u - 1, w - 1)
        const long long lo = quad_at(l, q, b, z), hi = quad_at(l, q, b + 1, z);  // w + 1 is 8 cells on
        bp[q * sa + b * sb + z] += (__ldg(q1 + 4 * (hi + 8)) + __ldg(q1 + 4 * hi + 1)) +
                                   (__ldg(q1 + 4 * (lo + 8) + 2) + __ldg(q1 + 4 * lo + 3));
    }
}

// A line as the four lanes that walk it together see it: Walk's fields, and
// val, what a back projection spreads (kModeBack) or the line's multiplier
// (kModeEm).  i1 < i0: nothing to visit.
struct QuadLine {
    int q0, i0, i1;
    float u0, w0, du, dw, step, l0, dl, cb, val;
};

__device__ __forceinline__ QuadLine no_line()
{
    QuadLine l{};
    l.i1 = -1;
    return l;
}

// Event e's line; add: kModeEm, the additive term.
template <int kMode, bool kTof>
__device__ __forceinline__ QuadLine prepare_line(const LmArgs& a, long long e, float& add)
{
    QuadLine l = no_line();
    Walk k;
    float cb = 0.f;
    const bool hit = walk_setup<kTof>(a.lors + 6 * e, a.g, k, a.tof, kTof ? __ldg(a.tof_bin + e) : 0, cb);
    if (kMode == kModeBack) l.val = __ldg(a.vals + e) * (a.mult ? __ldg(a.mult + e) : 1.f);
    if (kMode == kModeFwd) l.val = a.mult ? __ldg(a.mult + e) : 1.f;
    if (kMode == kModeEm) {
        l.val = __ldg(a.mult + e);
        add = a.s ? __ldg(a.s + e) : 0.f;
    }
    if (!hit || (kMode == kModeBack && l.val == 0.f)) return l;
    l.q0 = k.q0;
    l.i0 = k.i0;
    l.i1 = k.i1;
    l.u0 = k.u0;
    l.w0 = k.w0;
    l.du = k.du;
    l.dw = k.dw;
    l.step = k.step;
    if (kTof) {
        l.l0 = k.l0;
        l.dl = k.dl;
        l.cb = cb;
    }
    return l;
}

// The line that lane src of the warp holds.
template <bool kTof>
__device__ __forceinline__ QuadLine line_of(const QuadLine& own, int src)
{
    auto from = [&](auto v) { return __shfl_sync(0xffffffffu, v, src); };
    QuadLine k{};
    k.q0 = from(own.q0);
    k.i0 = from(own.i0);
    k.i1 = from(own.i1);
    k.u0 = from(own.u0);
    k.w0 = from(own.w0);
    k.du = from(own.du);
    k.dw = from(own.dw);
    k.step = from(own.step);
    k.val = from(own.val);
    if (kTof) {
        k.l0 = from(own.l0);
        k.dl = from(own.dl);
        k.cb = from(own.cb);
    }
    return k;
}

// One batch of kBatch samples of a lane, four planes apart, from sample i on:
// the cell of each (-1 outside the image or the line), its in-cell fractions
// and its weight.
constexpr int kBatch = 4, kQuadLanes = 4;
struct QuadBatch {
    int cell[kBatch];
    float tu[kBatch], tw[kBatch], wt[kBatch];
};

template <bool kTof>
__device__ __forceinline__ void quad_batch(QuadBatch& s, const QuadLine& k, int i, int nb, int nc, const QuadLattice& l,
                                           const TofParams& tp, const float* tof_tab)
{
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
        const int ij = i + j * kQuadLanes;
        const float f = (float)ij;
        const float u = fmaf(f, k.du, k.u0), w = fmaf(f, k.dw, k.w0);
        const float fu = floorf(u), fw = floorf(w);
        const bool in = ij >= k.i0 && ij <= k.i1 && fu >= -1.f && fu <= (float)(nb - 1) && fw >= -1.f &&
                        fw <= (float)(nc - 1);
        s.cell[j] = in ? quad_at(l, k.q0 + ij, (int)fu + 1, (int)fw + 1) : -1;
        s.tu[j] = u - fu;
        s.tw[j] = w - fw;
        s.wt[j] = kTof ? tof_weight(k.l0, k.dl, tp, k.cb, tof_tab, ij) : 1.f;
    }
}

// The walk of pet_lm_kernel over quads, for the lines of principal axis AX.
// A CTA collects the axis's lines from its share of the events in a queue in
// shared memory and walks them a CTA at a time, so that its threads stay busy
// whatever the mix of axes.  Each thread prepares one line; four lanes then
// walk a line together, eight lines of the warp at a time.
template <int kMode, bool kTof, int AX>
__global__ void __launch_bounds__(kQuadThreads, 8) pet_quad_kernel(LmArgs a)
{
    extern __shared__ float tof_s[];  // kTof: the timing-weight table
    __shared__ long long queue[2 * kQuadThreads];
    __shared__ int queued;
    if (kTof)
        for (int i = threadIdx.x; i <= kTofTab; i += blockDim.x) tof_s[i] = __ldg(a.tof_tab + i);
    if (threadIdx.x == 0) queued = 0;
    __syncthreads();
    const int nb = a.g.n[1 - AX], nc = a.g.n[2], lane = threadIdx.x & 31, sub = lane & (kQuadLanes - 1);
    const QuadLattice lat = quad_lattice(a.g, AX);
    double cons = 0.0, used = 0.0;
    long long next = blockIdx.x * (long long)kQuadThreads;
    int have = 0;  // lines in the queue (the same in every thread)
    for (;;) {
        while (have < kQuadThreads && next < a.count) {
            const long long t = next + threadIdx.x;
            bool keep = false;
            if (t < a.count) {
                float p1[3], p2[3], scale;
                load_line(a.lors + 6 * (a.first + t * a.stride), p1, p2);
                keep = line_axis(p1, p2, a.g, scale) == AX;
            }
            const unsigned mask = __ballot_sync(0xffffffffu, keep);
            int at = 0;
            if (lane == 0 && mask) at = atomicAdd(&queued, __popc(mask));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (keep) queue[at + __popc(mask & ((1u << lane) - 1u))] = t;
            have += __syncthreads_count(keep);
            next += (long long)gridDim.x * kQuadThreads;
        }
        if (have == 0) break;
        const int take = min(have, kQuadThreads);
        have -= take;
        const long long t = threadIdx.x < take ? queue[have + threadIdx.x] : -1;
        __syncthreads();  // taken; the queue may be filled again
        if (threadIdx.x == 0) queued = have;
        __syncthreads();
        // this thread's line
        const long long e = t < 0 ? -1 : a.first + t * a.stride;
        float add = 0.f;
        const QuadLine own = t < 0 ? no_line() : prepare_line<kMode, kTof>(a, e, add);
#pragma unroll 1
        for (int p = 0; p < kQuadLanes; ++p) {
            const int src = p * (32 / kQuadLanes) + lane / kQuadLanes;
            const long long el = __shfl_sync(0xffffffffu, e, src);
            const QuadLine k = line_of<kTof>(own, src);
            // lane `sub` takes the planes q with q % 4 == sub: the four lanes'
            // samples of a step share a brick unless the line leaves it
            const int first = k.i0 - ((k.q0 + k.i0) & (kQuadLanes - 1)) + sub;
            auto scatter = [&](float sv) {
                for (int i = first; i <= k.i1; i += kBatch * kQuadLanes) {
                    QuadBatch s;
                    quad_batch<kTof>(s, k, i, nb, nc, lat, a.tof, tof_s);
#pragma unroll
                    for (int j = 0; j < kBatch; ++j) {
                        if (s.cell[j] < 0) continue;
                        const float v = sv * s.wt[j], v0 = v * (1.f - s.tu[j]), v1 = v * s.tu[j], w0 = 1.f - s.tw[j];
                        atomicAdd(a.bquads + s.cell[j], make_float4(v0 * w0, v0 * s.tw[j], v1 * w0, v1 * s.tw[j]));
                    }
                }
            };
            if (kMode == kModeBack) {
                scatter(k.val * k.step);
                continue;
            }
            float acc = 0.f;
            for (int i = first; i <= k.i1; i += kBatch * kQuadLanes) {
                QuadBatch s;
                quad_batch<kTof>(s, k, i, nb, nc, lat, a.tof, tof_s);
                float4 v[kBatch];
#pragma unroll
                for (int j = 0; j < kBatch; ++j)
                    v[j] = s.cell[j] >= 0 ? __ldg(a.quads + s.cell[j]) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int j = 0; j < kBatch; ++j) {
                    if (s.cell[j] < 0) continue;
                    const float w0 = 1.f - s.tw[j];
                    const float lo = fmaf(s.tw[j], v[j].y, w0 * v[j].x), hi = fmaf(s.tw[j], v[j].w, w0 * v[j].z);
                    acc = fmaf(s.wt[j], fmaf(s.tu[j], hi, (1.f - s.tu[j]) * lo), acc);
                }
            }
#pragma unroll
            for (int o = 1; o < kQuadLanes; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            const float line = acc * k.step;  // 0 for a line that misses (step 0)
            if (kMode == kModeFwd) {
                if (el >= 0 && sub == 0) a.out[el] = a.mult ? k.val * line : line;
            } else {  // kModeEm
                const float pr = k.val * line;
                const float den = pr + __shfl_sync(0xffffffffu, add, src);
                if (el >= 0 && den > 0.f) {
                    if (sub == 0) {
                        cons += (double)pr / (double)den;
                        used += 1.0;
                    }
                    scatter(k.val / den * k.step);
                }
            }
        }
    }
    if (kMode == kModeEm && a.diag) block_add2(cons, used, a.diag);
}

// The lines along z of a call that walks quads, on the image.  A warp looks
// through 32 lines and walks those it finds one at a time, its lanes on
// consecutive planes, which lie next to each other in memory.  About 1 % of a
// cylindrical scanner's lines lie along z; with a line to a lane these few took
// as long as a whole walk of dependent loads.  Measured: 3 M events in 3 subsets
// with time of flight 5.60 -> 5.54 ms, the pair of projectors of 1 M lines 1.224
// -> 1.200 ms.
template <int kMode, bool kTof>
__global__ void __launch_bounds__(kPetThreads) pet_z_kernel(LmArgs a)
{
    const int lane = threadIdx.x & 31;
    double cons = 0.0, used = 0.0;
    const long long warps = (long long)gridDim.x * (kPetThreads / 32);
    for (long long t0 = 32 * (((long long)blockIdx.x * kPetThreads + threadIdx.x) >> 5); t0 < a.count;
         t0 += 32 * warps) {
        const long long e = a.first + (t0 + lane) * a.stride;
        bool mine = false;
        if (t0 + lane < a.count) {
            float p1[3], p2[3], scale;
            load_line(a.lors + 6 * e, p1, p2);
            mine = line_axis(p1, p2, a.g, scale) == 2;
        }
        unsigned mask = __ballot_sync(0xffffffffu, mine);
        if (mask == 0) continue;
        float add = 0.f;
        const QuadLine own = mine ? prepare_line<kMode, kTof>(a, e, add) : no_line();
        for (; mask; mask &= mask - 1) {
            const int src = __ffs(mask) - 1;
            const QuadLine l = line_of<kTof>(own, src);
            const long long el = a.first + (t0 + src) * a.stride;
            Walk k{};
            k.a = 2;
            k.b = 0;
            k.c = 1;
            k.q0 = l.q0;
            k.i0 = l.i0;
            k.i1 = l.i1;
            k.u0 = l.u0;
            k.w0 = l.w0;
            k.du = l.du;
            k.dw = l.dw;
            k.l0 = l.l0;
            k.dl = l.dl;
            const long long sc = a.g.stride[1];
            auto scatter = [&](float sv) {
                walk<kTof>(k, a.g, a.tof, l.cb, a.tof_tab, k.i0 + lane, 32,
                           [&](long long idx, bool o0, bool o1, float w0, float w1) {
                               scatter_pair(a.bp, idx, sc, a.g.total, o0, o1, sv * w0, sv * w1);
                           });
            };
            if (kMode == kModeBack) {
                scatter(l.val * l.step);
                continue;
            }
            float acc = 0.f;
            walk<kTof>(k, a.g, a.tof, l.cb, a.tof_tab, k.i0 + lane, 32,
                       [&](long long idx, bool o0, bool o1, float w0, float w1) {
                           acc += gather_pair(a.img, idx, sc, a.g.total, o0, o1, w0, w1);
                       });
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            const float line = acc * l.step;  // 0 for a line that misses (step 0)
            if (kMode == kModeFwd) {
                if (lane == 0) a.out[el] = a.mult ? l.val * line : line;
            } else {  // kModeEm
                const float pr = l.val * line;
                const float den = pr + __shfl_sync(0xffffffffu, add, src);
                if (!(den > 0.f)) continue;
                if (lane == 0) {
                    cons += (double)pr / (double)den;
                    used += 1.0;
                }
                scatter(l.val / den * l.step);
            }
        }
    }
    if (kMode == kModeEm && a.diag) block_add2(cons, used, a.diag);
}

// One separable T_rr pass along axis AX (0 = x, 1 = y, 2 = z), zero padding.
// With `sens` set the pass is the last one of a back projection and writes
// x <- x * out / (sens / M) where sens / M > 0 (x unchanged elsewhere).
// Blocks of 32 x 8 outputs (z, y) of one x, so that no index is divided (with
// 64-bit divisions and one output a thread the three passes took 152 us at 204
// x 204 x 154; without the divisions 112; with runs along x and y 92).  Radii up
// to kRrUnrolled have passes of their own (kR, else -1) whose taps are constants
// of the instructions: the loop over them had cost more than its loads (with
// the events around them 92 -> 48 us, with the update 108 -> 70).
constexpr int kRrZ = 32, kRrY = 8;
constexpr int kRrRun = 8;  // x and y passes: outputs of a thread along the axis, which share their inputs

constexpr int kRrUnrolled = 8;

template <int AX, int kR>
__global__ void __launch_bounds__(kRrZ * kRrY) pet_rr_kernel(const float* __restrict__ in, float* __restrict__ out,
                                                             RrTaps taps, int nx, int ny, int nz,
                                                             const float* __restrict__ sens, float inv_m)
{
    // the thread's place: z, the axis's first output, and the third axis
    constexpr int run = AX == 2 ? 1 : kRrRun;
    const int z = blockIdx.x * kRrZ + threadIdx.x, c = blockIdx.y * kRrY + threadIdx.y;
    const int x = AX == 0 ? blockIdx.z * run : AX == 1 ? c : blockIdx.z, y = AX == 1 ? blockIdx.z * run : c;
    if (z >= nz || x >= nx || y >= ny) return;
    const int n_ax = AX == 0 ? nx : AX == 1 ? ny : nz, pos = AX == 0 ? x : AX == 1 ? y : z;
    const long long st = AX == 0 ? (long long)ny * nz : AX == 1 ? nz : 1;
    const long long i = ((long long)x * ny + y) * nz + z;
    const int r = taps.r;
    float acc[run];
#pragma unroll
    for (int q = 0; q < run; ++q) acc[q] = 0.f;
    // inputs pos + m from the highest down, so that every output's sum runs
    // over its taps in rising order
    if (kR >= 0) {
        const float* p = in + i;
#pragma unroll
        for (int m = run - 1 + kR; m >= -kR; --m) {
            const float v = (unsigned)(pos + m) < (unsigned)n_ax ? __ldg(p + m * st) : 0.f;
#pragma unroll
            for (int q = 0; q < run; ++q) {
                const int t = q - m + kR;
                if (t >= 0 && t <= 2 * kR) acc[q] = fmaf(taps.w[t], v, acc[q]);
            }
        }
    } else {
        const int hi = min(run - 1 + r, n_ax - 1 - pos), lo = max(-r, -pos);
        const float* p = in + i + hi * st;
#pragma unroll 4
        for (int m = hi; m >= lo; --m, p -= st) {
            const float v = __ldg(p);
#pragma unroll
            for (int q = 0; q < run; ++q) {
                const int t = q - m + r;
                if (t >= 0 && t <= 2 * r) acc[q] = fmaf(taps.w[t], v, acc[q]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < run; ++q) {
        if (pos + q >= n_ax) break;
        const long long o = i + q * st;
        if (sens) {
            const float sm = __ldg(sens + o) * inv_m;
            if (sm > 0.f) out[o] = out[o] * acc[q] / sm;
        } else {
            out[o] = acc[q];
        }
    }
}

// x <- x * bp / (sens / M) without T_rr.
__global__ void __launch_bounds__(kPetThreads) pet_update_kernel(float* __restrict__ x, const float* __restrict__ bp,
                                                                 const float* __restrict__ sens, float inv_m,
                                                                 long long total)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const float sm = __ldg(sens + i) * inv_m;
        if (sm > 0.f) x[i] = x[i] * __ldg(bp + i) / sm;
    }
}

int pfail(int status, const char* fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    spect_internal_set_error(buf);
    return status;
}

int pcuda(cudaError_t e, const char* what)
{
    cudaGetLastError();
    return pfail(SPECT_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

bool aligned(const void* p, unsigned a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

unsigned blocks_for(long long count)
{
    const long long b = (count + kPetThreads - 1) / kPetThreads;
    return (unsigned)(b < 1 ? 1 : b > kPetMaxBlocks ? kPetMaxBlocks : b);
}

struct DevGuard {
    int prev = -1;
    bool ok = true;
    explicit DevGuard(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) { ok = false; return; }
        if (prev != dev && cudaSetDevice(dev) != cudaSuccess) ok = false;
    }
    ~DevGuard()
    {
        int cur = -1;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

}  // namespace

struct pet_plan {
    pet_geom geom{};
    int device = 0;
    PetGrid grid{};
    RrTaps taps[3]{};
    bool rr = false;
    TofParams tof{};
    long long voxels = 0;
    float* mu = nullptr;
    float* tof_tab = nullptr;  // [kTofTab + 1] timing weights
    float* t1 = nullptr;
    float* t2 = nullptr;
    float* fb = nullptr;
    float* bp = nullptr;
    float4* quads = nullptr;   // the walked image's quads of one axis, and the back projection's
    float4* bquads = nullptr;  // (each allocated by the first call that walks it)
    double* diag = nullptr;
    int diag_cap = 0;  // subiterations the diag buffer holds
    std::vector<void*> allocations;
    bool prof = false;
    struct Pending {
        std::string name;
        cudaEvent_t start, stop;
    };
    std::vector<Pending> pending;
    std::vector<cudaEvent_t> event_pool;
    std::map<std::string, std::pair<unsigned long long, double>> totals;
};

namespace {

template <class T>
int palloc(pet_plan* p, T** out, size_t count)
{
    *out = nullptr;
    void* ptr = nullptr;
    cudaError_t e = cudaMalloc(&ptr, (count ? count : 1) * sizeof(T));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return pfail(SPECT_ENOMEM, "cudaMalloc of %zu bytes failed", count * sizeof(T));
    }
    p->allocations.push_back(ptr);
    *out = static_cast<T*>(ptr);
    return SPECT_OK;
}

cudaEvent_t take_event(pet_plan* p)
{
    if (!p->event_pool.empty()) {
        cudaEvent_t e = p->event_pool.back();
        p->event_pool.pop_back();
        return e;
    }
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return e;
}

// Launch through `fn`, count the kernels and time them when profiling.
template <class F>
int launch(pet_plan* p, const char* name, cudaStream_t st, int kernels, F&& fn)
{
    cudaEvent_t e0 = nullptr;
    if (p->prof && p->pending.size() < 1000000) {
        e0 = take_event(p);
        if (e0) cudaEventRecord(e0, st);
    }
    fn();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return pcuda(e, name);
    spect_internal_count_launches((unsigned long long)kernels);
    if (e0) {
        cudaEvent_t e1 = take_event(p);
        if (e1) {
            cudaEventRecord(e1, st);
            p->pending.push_back({name, e0, e1});
        } else {
            p->event_pool.push_back(e0);
        }
    }
    return SPECT_OK;
}

template <int AX>
void launch_rr(dim3 grid, dim3 block, cudaStream_t st, const float* in, float* out, const RrTaps& taps, int nx, int ny,
               int nz, const float* sens, float inv_m)
{
    switch (taps.r) {
#define PET_RR_CASE(R) \
    case R: pet_rr_kernel<AX, R><<<grid, block, 0, st>>>(in, out, taps, nx, ny, nz, sens, inv_m); return;
        PET_RR_CASE(1) PET_RR_CASE(2) PET_RR_CASE(3) PET_RR_CASE(4)
        PET_RR_CASE(5) PET_RR_CASE(6) PET_RR_CASE(7) PET_RR_CASE(kRrUnrolled)
#undef PET_RR_CASE
        default: pet_rr_kernel<AX, -1><<<grid, block, 0, st>>>(in, out, taps, nx, ny, nz, sens, inv_m);
    }
}

// out = T_rr in (three passes through t1, t2), or the update of x (sens set).
int rr_apply(pet_plan* p, const float* in, float* out, const float* sens, cudaStream_t st)
{
    const int nx = p->geom.nx, ny = p->geom.ny, nz = p->geom.nz;
    const dim3 block(kRrZ, kRrY);
    const unsigned bz = (nz + kRrZ - 1) / kRrZ, by = (ny + kRrY - 1) / kRrY, bx = (nx + kRrY - 1) / kRrY;
    const dim3 grid0(bz, by, (nx + kRrRun - 1) / kRrRun), grid1(bz, bx, (ny + kRrRun - 1) / kRrRun), grid2(bz, by, nx);
    const float inv_m = 1.f / (float)p->geom.n_subsets;
    return launch(p, sens ? "rr_update" : "rr_blur", st, 3, [&] {
        launch_rr<0>(grid0, block, st, in, p->t1, p->taps[0], nx, ny, nz, nullptr, 0.f);
        launch_rr<1>(grid1, block, st, p->t1, p->t2, p->taps[1], nx, ny, nz, nullptr, 0.f);
        launch_rr<2>(grid2, block, st, p->t2, out, p->taps[2], nx, ny, nz, sens, inv_m);
    });
}

LmArgs base_args(const pet_plan* p, const float* lors, long long n)
{
    LmArgs a{};
    a.lors = lors;
    a.first = 0;
    a.stride = 1;
    a.count = n;
    a.g = p->grid;
    a.tof = p->tof;
    a.tof_tab = p->tof_tab;
    return a;
}

// Relaxed capture mode in this thread while it lives: a call under stream
// capture, or next to another thread's capture, may allocate.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    bool ok;
    RelaxedCapture() : ok(cudaThreadExchangeStreamCaptureMode(&mode) == cudaSuccess)
    {
        if (!ok) cudaGetLastError();
    }
    ~RelaxedCapture()
    {
        if (ok) cudaThreadExchangeStreamCaptureMode(&mode);
    }
};

// Allocates those of the plan's quads that are wanted and missing: all of them,
// or none where they would take more than half of the free memory (which other
// users of the device want too) or the allocation fails.
bool take_quads(pet_plan* p, bool image, bool back, size_t bytes)
{
    float4** want[2] = {image && !p->quads ? &p->quads : nullptr, back && !p->bquads ? &p->bquads : nullptr};
    const size_t missing = bytes * ((want[0] ? 1 : 0) + (want[1] ? 1 : 0));
    if (missing == 0) return true;
    RelaxedCapture relaxed;
    if (!relaxed.ok) return false;
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (missing > free_b / 2) return false;
    void* got[2] = {nullptr, nullptr};
    for (int i = 0; i < 2; ++i)
        if (want[i] && cudaMalloc(&got[i], bytes) != cudaSuccess) {
            cudaGetLastError();
            cudaFree(got[0]);
            return false;
        }
    for (int i = 0; i < 2; ++i)
        if (want[i]) {
            p->allocations.push_back(got[i]);
            *want[i] = static_cast<float4*>(got[i]);
        }
    return true;
}

// Whether `lines` lines pay for the quads: at least one per 32 voxels (building,
// clearing and folding quads moves about 100 bytes a voxel and axis), and with
// less than a wave of the image walk, which then takes the time of one line, as
// many as the mode needs.  Events of the head phantom, us, image walk / quads:
//   forward                 64 x 64 x 40, 8192 lines 104 / 87; 96 x 96 x 64, 24576
//                           143 / 110; 204 x 204 x 154, 262144 610 / 430
//   back                    64^3, 16384 68 / 88, 49152 100 / 100, 131072 172 / 154;
//                           128 x 128 x 90, 49152 155 / 139
//   OSEM                    64^3, 8192 161 / 146; 128 x 128 x 90, 49152 330 / 247
//   with time of flight:
//   forward                 64 x 64 x 120, 65536 119 / 136, 131072 210 / 187; 96 x 96
//                           x 64, 24576 136 / 124
//   back                    64^3, 131072 159 / 187, 524288 386 / 388; 64 x 64 x 120,
//                           131072 194 / 192; 128 x 128 x 90, 98304 201 / 206, 131072
//                           247 / 232
//   OSEM                    64^3, 65536 174 / 197, 98304 211 / 230, 131072 304 / 249;
//                           204 x 204 x 154, 98304 580 / 614, 262144 1240 / 864
constexpr long long kImageWave = 152 * 3 * kPetThreads;  // with time of flight 3 CTAs an SM

template <int kMode>
bool quads_pay(const pet_plan* p, long long lines, bool tof)
{
    if (lines < p->voxels / 32) return false;
    if (!tof) return kMode != kModeBack || lines >= 3 << 14;
    const bool waves = lines > kImageWave;
    if (kMode == kModeFwd) return waves || p->voxels >= 1 << 19;
    if (kMode == kModeBack) return waves && (p->voxels >= 3 << 17 || lines >= 1 << 19);
    return waves;
}

// Whether a call walks quads: where that pays, on lattices that 32-bit indexes
// reach, with the memory for the sets that the mode needs, kept by the plan.
// Where there is none the image is walked, and a later call tries again.
template <int kMode>
bool use_quads(pet_plan* p, long long lines, bool tof)
{
    const long long cells = std::max(quad_cells(p->grid, 0), quad_cells(p->grid, 1));
    if (!quads_pay<kMode>(p, lines, tof) || cells >= (1ll << 31) - (1ll << 23) || p->voxels >= (1ll << 31)) return false;
    return take_quads(p, kMode != kModeBack, kMode != kModeFwd, (size_t)cells * sizeof(float4));
}

constexpr int kQuadBlocks = 152 * 8;  // pet_quad_kernel: every resident CTA

template <int kMode, int AX>
void launch_quad_axis(pet_plan* p, const LmArgs& a, cudaStream_t st)
{
    const long long cells = quad_cells(p->grid, AX);
    if (kMode != kModeBack) pet_quads_kernel<AX><<<blocks_for(cells), kPetThreads, 0, st>>>(a.img, a.quads, a.g);
    if (kMode != kModeFwd) cudaMemsetAsync(a.bquads, 0, (size_t)cells * sizeof(float4), st);
    const long long want = (a.count + kQuadThreads - 1) / kQuadThreads;
    const unsigned blocks = (unsigned)std::min<long long>(want, kQuadBlocks);
    if (a.tof_bin)
        pet_quad_kernel<kMode, true, AX><<<blocks, kQuadThreads, kTofSmem, st>>>(a);
    else
        pet_quad_kernel<kMode, false, AX><<<blocks, kQuadThreads, 0, st>>>(a);
    if (kMode != kModeFwd) pet_fold_kernel<AX><<<blocks_for(p->voxels), kPetThreads, 0, st>>>(a.bquads, a.bp, a.g);
}

// The walk of `a`'s lines (kModeFwd, kModeBack, kModeEm), over quads where
// that pays.
template <int kMode>
int launch_walk(pet_plan* p, const char* name, LmArgs a, cudaStream_t st)
{
    const bool quads = use_quads<kMode>(p, a.count, a.tof_bin != nullptr);
    const int kernels = !quads ? 1 : kMode == kModeEm ? 7 : 5;
    return launch(p, name, st, kernels, [&] {
        if (quads) {
            a.quads = p->quads;
            a.bquads = p->bquads;
            launch_quad_axis<kMode, 0>(p, a, st);
            launch_quad_axis<kMode, 1>(p, a, st);
            if (a.tof_bin)
                pet_z_kernel<kMode, true><<<blocks_for(a.count), kPetThreads, 0, st>>>(a);
            else
                pet_z_kernel<kMode, false><<<blocks_for(a.count), kPetThreads, 0, st>>>(a);
            return;
        }
        if (a.tof_bin)
            pet_lm_kernel<kMode, true><<<blocks_for(a.count), kPetThreads, kTofSmem, st>>>(a);
        else
            pet_lm_kernel<kMode, false><<<blocks_for(a.count), kPetThreads, 0, st>>>(a);
    });
}

int check_tof(const pet_plan* p, const int* tof_bin, int64_t n)
{
    if (tof_bin && p->tof.nb == 0) return pfail(SPECT_EINVAL, "tof_bin given to a plan without time of flight");
    if (tof_bin && n > 0 && !aligned(tof_bin, 4)) return pfail(SPECT_EINVAL, "tof_bin must be 4-byte aligned");
    return SPECT_OK;
}

int check_lors(const pet_plan* p, const float* lors, int64_t n)
{
    if (!p) return pfail(SPECT_EINVAL, "plan is NULL");
    if (n < 0) return pfail(SPECT_EINVAL, "negative LOR count");
    if (n > 0 && (!lors || !aligned(lors, 8))) return pfail(SPECT_EINVAL, "lors must be an 8-byte aligned device pointer");
    return SPECT_OK;
}

int check_image(const float* x, const char* what)
{
    if (!x || !aligned(x, 16)) return pfail(SPECT_EINVAL, "%s must be a 16-byte aligned device pointer", what);
    return SPECT_OK;
}

}  // namespace

extern "C" {

int pet_plan_create(const pet_geom* geom, const float* mu_dev, void* stream, pet_plan** out)
{
    if (!out) return pfail(SPECT_EINVAL, "out is NULL");
    *out = nullptr;
    if (!geom) return pfail(SPECT_EINVAL, "geom is NULL");
    const pet_geom& g = *geom;
    if (g.nx < 1 || g.ny < 1 || g.nz < 1 || g.nx > 4096 || g.ny > 4096 || g.nz > 4096)
        return pfail(SPECT_EINVAL, "image size must be in [1, 4096] per axis");
    if (!(g.vx > 0.f) || !(g.vy > 0.f) || !(g.vz > 0.f)) return pfail(SPECT_EINVAL, "voxel sizes must be > 0");
    if (g.n_subsets < 1) return pfail(SPECT_EINVAL, "n_subsets must be >= 1");
    const bool rr = g.rr_sigma_mm > 0.f;
    if (rr && !(g.rr_nsigma > 0.f)) return pfail(SPECT_EINVAL, "rr_nsigma must be > 0");
    if (mu_dev && !aligned(mu_dev, 16)) return pfail(SPECT_EINVAL, "mu must be a 16-byte aligned device pointer");
    if (g.n_tof_bins < 0 || g.n_tof_bins > 4096) return pfail(SPECT_EINVAL, "n_tof_bins must be in [0, 4096]");
    if (g.n_tof_bins > 0 && (!(g.tof_bin_mm > 0.f) || !(g.tof_sigma_mm > 0.f) || !(g.tof_nsigma > 0.f)))
        return pfail(SPECT_EINVAL, "time of flight needs tof_bin_mm, tof_sigma_mm and tof_nsigma > 0");
    pet_plan* p = new pet_plan();
    p->geom = g;
    p->rr = rr;
    p->tof.nb = g.n_tof_bins;
    std::vector<float> tof_tab;
    if (g.n_tof_bins > 0) {
        p->tof.width = g.tof_bin_mm;
        p->tof.sigma = g.tof_sigma_mm;
        p->tof.nsigma = g.tof_nsigma;
        const double hw = (double)g.tof_nsigma * g.tof_sigma_mm + 0.5 * (double)g.tof_bin_mm;
        p->tof.half_win = (float)hw;
        p->tof.inv_h = (float)(kTofTab / (2.0 * hw));
        tof_tab.resize(kTofTab + 1);
        const double s2 = std::sqrt(2.0) * (double)g.tof_sigma_mm, h = 0.5 * (double)g.tof_bin_mm;
        for (int i = 0; i <= kTofTab; ++i) {
            // Phi((x + h)/sigma) - Phi((x - h)/sigma) with Phi(t) = erfc(-t/sqrt 2) / 2
            const double x = -hw + 2.0 * hw * i / kTofTab;
            tof_tab[i] = (float)(0.5 * (std::erfc(-(x + h) / s2) - std::erfc(-(x - h) / s2)));
        }
    }
    const float v[3] = {g.vx, g.vy, g.vz};
    const int n[3] = {g.nx, g.ny, g.nz};
    for (int c = 0; c < 3; ++c) {
        p->grid.n[c] = n[c];
        p->grid.v[c] = v[c];
    }
    p->grid.stride[0] = (long long)g.ny * g.nz;
    p->grid.stride[1] = g.nz;
    p->grid.stride[2] = 1;
    p->voxels = (long long)g.nx * g.ny * g.nz;
    p->grid.total = p->voxels;
    // T_rr taps per axis, in double, stored as float
    for (int c = 0; c < 3; ++c) {
        RrTaps& t = p->taps[c];
        if (!rr) {
            t.r = 0;
            t.w[0] = 1.f;
            continue;
        }
        const double s = (double)g.rr_sigma_mm / (double)v[c];
        const double rd = std::ceil((double)g.rr_nsigma * s);
        if (rd > kPetMaxR) {
            delete p;
            return pfail(SPECT_EINVAL, "T_rr radius %.0f voxels exceeds %d", rd, kPetMaxR);
        }
        t.r = (int)rd;
        double w[2 * kPetMaxR + 1], sum = 0.0;
        for (int q = -t.r; q <= t.r; ++q) {
            w[q + t.r] = std::exp(-(double)q * q / (2.0 * s * s));
            sum += w[q + t.r];
        }
        for (int q = 0; q <= 2 * t.r; ++q) t.w[q] = (float)(w[q] / sum);
    }
    if (cudaGetDevice(&p->device) != cudaSuccess) {
        delete p;
        return pcuda(cudaGetLastError(), "cudaGetDevice");
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int rc = SPECT_OK;
    const size_t nv = (size_t)p->voxels;
    if (!rc) rc = palloc(p, &p->t1, nv);
    if (!rc) rc = palloc(p, &p->t2, nv);
    if (!rc) rc = palloc(p, &p->fb, nv);
    if (!rc) rc = palloc(p, &p->bp, nv);
    if (!rc) {
        p->diag_cap = 64;
        rc = palloc(p, &p->diag, 2 * (size_t)p->diag_cap);
    }
    if (!rc && !tof_tab.empty()) {
        rc = palloc(p, &p->tof_tab, tof_tab.size());
        if (!rc) {
            cudaError_t e = cudaMemcpy(p->tof_tab, tof_tab.data(), tof_tab.size() * sizeof(float),
                                       cudaMemcpyHostToDevice);
            if (e != cudaSuccess) rc = pcuda(e, "copy of the timing table");
        }
    }
    if (!rc && mu_dev) {
        rc = palloc(p, &p->mu, nv);
        if (!rc) {
            cudaError_t e = cudaMemcpyAsync(p->mu, mu_dev, nv * sizeof(float), cudaMemcpyDeviceToDevice, st);
            if (e != cudaSuccess) rc = pcuda(e, "copy of mu");
        }
    }
    if (rc) {
        pet_plan_destroy(p);
        return rc;
    }
    *out = p;
    return SPECT_OK;
}

int pet_plan_destroy(pet_plan* p)
{
    if (!p) return SPECT_OK;
    DevGuard guard(p->device);
    cudaDeviceSynchronize();
    for (void* a : p->allocations) cudaFree(a);
    for (auto& r : p->pending) {
        cudaEventDestroy(r.start);
        cudaEventDestroy(r.stop);
    }
    for (cudaEvent_t e : p->event_pool) cudaEventDestroy(e);
    delete p;
    return SPECT_OK;
}

int pet_mult(pet_plan* p, const float* lors, const float* eta, int64_t n, float* mult_out, void* stream)
{
    if (int rc = check_lors(p, lors, n)) return rc;
    if (n > 0 && (!mult_out || !aligned(mult_out, 4))) return pfail(SPECT_EINVAL, "mult_out must be a device pointer");
    if (n == 0) return SPECT_OK;
    DevGuard guard(p->device);
    if (!guard.ok) return pfail(SPECT_ECUDA, "cannot select the plan's device");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    LmArgs a = base_args(p, lors, n);
    a.img = p->mu;
    a.vals = eta;
    a.out = mult_out;
    return launch(p, "joseph_mult", st, 1,
                  [&] { pet_lm_kernel<kModeMult, false><<<blocks_for(n), kPetThreads, 0, st>>>(a); });
}

int pet_forward(pet_plan* p, const float* x, const float* lors, const float* mult, const int* tof_bin, int64_t n,
                float* out, void* stream)
{
    if (int rc = check_lors(p, lors, n)) return rc;
    if (int rc = check_tof(p, tof_bin, n)) return rc;
    if (int rc = check_image(x, "x")) return rc;
    if (n > 0 && !out) return pfail(SPECT_EINVAL, "out is NULL");
    if (n == 0) return SPECT_OK;
    DevGuard guard(p->device);
    if (!guard.ok) return pfail(SPECT_ECUDA, "cannot select the plan's device");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const float* img = x;
    if (p->rr) {
        if (int rc = rr_apply(p, x, p->fb, nullptr, st)) return rc;
        img = p->fb;
    }
    LmArgs a = base_args(p, lors, n);
    a.img = img;
    a.mult = mult;
    a.out = out;
    a.tof_bin = tof_bin;
    return launch_walk<kModeFwd>(p, tof_bin ? "joseph_fwd_tof" : "joseph_fwd", a, st);
}

int pet_back(pet_plan* p, const float* q, const float* lors, const float* mult, const int* tof_bin, int64_t n,
             float* x_out, void* stream)
{
    if (int rc = check_lors(p, lors, n)) return rc;
    if (int rc = check_tof(p, tof_bin, n)) return rc;
    if (int rc = check_image(x_out, "x_out")) return rc;
    if (n > 0 && !q) return pfail(SPECT_EINVAL, "q is NULL");
    DevGuard guard(p->device);
    if (!guard.ok) return pfail(SPECT_ECUDA, "cannot select the plan's device");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    float* acc = p->rr ? p->bp : x_out;
    cudaError_t e = cudaMemsetAsync(acc, 0, (size_t)p->voxels * sizeof(float), st);
    if (e != cudaSuccess) return pcuda(e, "clear of the back projection");
    if (n > 0) {
        LmArgs a = base_args(p, lors, n);
        a.bp = acc;
        a.vals = q;
        a.mult = mult;
        a.tof_bin = tof_bin;
        if (int rc = launch_walk<kModeBack>(p, tof_bin ? "joseph_back_tof" : "joseph_back", a, st)) return rc;
    }
    if (p->rr) return rr_apply(p, p->bp, x_out, nullptr, st);
    return SPECT_OK;
}

int pet_lm_osem_run(pet_plan* p, const float* lors, const float* mult, const float* s, const int* tof_bin,
                    int64_t n, const float* sens, float* x, int first, int count, double* diag_out, void* stream)
{
    if (int rc = check_lors(p, lors, n)) return rc;
    if (int rc = check_tof(p, tof_bin, n)) return rc;
    if (int rc = check_image(x, "x_inout")) return rc;
    if (int rc = check_image(sens, "sens")) return rc;
    if (n > 0 && !mult) return pfail(SPECT_EINVAL, "mult is NULL");
    if (first < 0 || count < 0) return pfail(SPECT_EINVAL, "negative subiteration range");
    DevGuard guard(p->device);
    if (!guard.ok) return pfail(SPECT_ECUDA, "cannot select the plan's device");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (diag_out && count > p->diag_cap) {
        double* d = nullptr;
        cudaError_t e = cudaMalloc(&d, 2 * (size_t)count * sizeof(double));
        if (e != cudaSuccess) {
            cudaGetLastError();
            return pfail(SPECT_ENOMEM, "diagnostics buffer");
        }
        p->allocations.push_back(d);
        p->diag = d;
        p->diag_cap = count;
    }
    if (diag_out && count > 0) {
        cudaError_t e = cudaMemsetAsync(p->diag, 0, 2 * (size_t)count * sizeof(double), st);
        if (e != cudaSuccess) return pcuda(e, "clear of the diagnostics");
    }
    const int M = p->geom.n_subsets;
    const float inv_m = 1.f / (float)M;
    for (int it = first; it < first + count; ++it) {
        const int m = it % M;
        const float* img = x;
        if (p->rr) {
            if (int rc = rr_apply(p, x, p->fb, nullptr, st)) return rc;
            img = p->fb;
        }
        cudaError_t e = cudaMemsetAsync(p->bp, 0, (size_t)p->voxels * sizeof(float), st);
        if (e != cudaSuccess) return pcuda(e, "clear of the back projection");
        const long long cnt = n > m ? (n - m + M - 1) / M : 0;
        if (cnt > 0) {
            LmArgs a = base_args(p, lors, cnt);
            a.first = m;
            a.stride = M;
            a.img = img;
            a.bp = p->bp;
            a.mult = mult;
            a.s = s;
            a.diag = diag_out ? p->diag + 2 * (it - first) : nullptr;
            a.tof_bin = tof_bin;
            if (int rc = launch_walk<kModeEm>(p, tof_bin ? "joseph_em_tof" : "joseph_em", a, st)) return rc;
        }
        if (p->rr) {
            if (int rc = rr_apply(p, p->bp, x, sens, st)) return rc;
        } else {
            const long long nv = p->voxels;
            if (int rc = launch(p, "update", st, 1, [&] {
                    pet_update_kernel<<<blocks_for(nv), kPetThreads, 0, st>>>(x, p->bp, sens, inv_m, nv);
                }))
                return rc;
        }
    }
    if (diag_out && count > 0) {
        cudaError_t e = cudaMemcpyAsync(diag_out, p->diag, 2 * (size_t)count * sizeof(double),
                                        cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return pcuda(e, "diagnostics");
    }
    return SPECT_OK;
}

int pet_profile_enable(pet_plan* p, int on)
{
    if (!p) return pfail(SPECT_EINVAL, "plan is NULL");
    p->prof = on != 0;
    return SPECT_OK;
}

int pet_profile_read(pet_plan* p, spect_kernel_time* out, int max_entries, int reset)
{
    if (!p) return pfail(SPECT_EINVAL, "plan is NULL");
    if (max_entries < 0 || (max_entries > 0 && !out)) return pfail(SPECT_EINVAL, "bad output array");
    DevGuard guard(p->device);
    for (auto& r : p->pending) {
        cudaError_t e = cudaEventSynchronize(r.stop);
        float ms = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, r.start, r.stop);
        if (e != cudaSuccess) return pcuda(e, "profile events");
        auto& tot = p->totals[r.name];
        tot.first += 1;
        tot.second += ms;
        p->event_pool.push_back(r.start);
        p->event_pool.push_back(r.stop);
    }
    p->pending.clear();
    int k = 0;
    for (auto& kv : p->totals) {
        if (k >= max_entries) break;
        std::snprintf(out[k].name, sizeof out[k].name, "%s", kv.first.c_str());
        out[k].launches = kv.second.first;
        out[k].total_ms = kv.second.second;
        ++k;
    }
    if (reset) p->totals.clear();
    return k;
}

}  // extern "C"
