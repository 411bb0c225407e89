// Host-side tiling and dispatch of the FP32 plane kernels.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"

namespace spect {

namespace {

int round_up(int v, int m) { return (v + m - 1) / m * m; }

// Forward z tile of ktile columns, its halo a multiple of `halo`; smem 0 where
// its strips do not fit.
PlaneTiling make_tiling(int n, int nz, int rmax, int ktile, int halo, size_t cap, size_t limit)
{
    PlaneTiling t{};
    t.ktile = ktile;
    t.ntiles = (nz + ktile - 1) / ktile;
    t.rh = round_up(rmax, t.ntiles > 1 ? halo : 2);
    t.ktpad = round_up(ktile, kStrip);
    t.npad = round_up(n, kStrip);
    t.sp = ((t.ktpad + 2 * t.rh) / 2) | 1;
    t.sq = ((t.npad + 2 * t.rh) / 2) | 1;
    // P and Q quads, the per-plane tap-row table (32 bytes per row) and the
    // two-plane tap buffer
    const size_t pq = 16 * ((size_t)(t.npad / 2) * t.sp + (size_t)(t.ktpad / 2) * t.sq);
    t.off_taps = (int)(pq + 32 * (size_t)n);
    t.smem = (size_t)t.off_taps + 2 * kTapRow * sizeof(float);
    // the attenuation buffer where it fits and a plane is one copy (a tile's
    // rows would be copied one by one, about 60 ns each)
    const size_t off = (t.smem + 15) & ~(size_t)15, end = off + (size_t)n * nz * sizeof(float);
    if (t.ntiles == 1 && end + 8 <= limit) {
        t.smem_a = true;
        t.off_a = (int)off;
        t.off_bar = (int)end;
        t.smem = end + 8;
    }
    // CTA size.  The staging and its latency scale with the warps, so a CTA
    // takes all the threads an SM holds, or half of them where two fit: at
    // least a thread per j-blur strip (ktpad/2 column pairs x npad/kStrip row
    // strips) where that is within the limit, else several strips per thread.
    // Measured (forward, one subset): 64^3 x 8 angles 4 x 128 threads 18.5 us,
    // 2 x 256 16.5, 1 x 512 18.4; 96^3 x 12 288 threads 48.9, 512 45.2;
    // 132 x 44 x 60 2 x 224 242, 1 x 320 375, 1 x 448 347.
    const int items = (t.ktpad / 2) * (t.npad / kStrip);
    const bool two = 2 * (t.smem + 1024) <= kSmSmem;
    t.threads = two && items <= kPlaneThreads / 2 ? kPlaneThreads / 2 : kPlaneThreads;
    t.ctas = two && t.threads <= kPlaneThreads / 2 ? 2 : 1;
    t.ipt = (items + t.threads - 1) / t.threads;
    t.high = rmax > kLowR || t.ipt > 1;
    if (t.ipt > kMaxIpt || (size_t)t.off_taps + 2 * kTapRow * sizeof(float) > cap) t.smem = 0;
    return t;
}

// Columns of the volume a tiling stages per plane (tile plus in-volume halo).
long staged_columns(const PlaneTiling& t, int nz)
{
    long cols = 0;
    for (int tile = 0; tile < t.ntiles; ++tile) {
        const int kw0 = tile * t.ktile - t.rh;
        cols += std::min(nz, kw0 + t.ktpad + 2 * t.rh) - std::max(0, kw0);
    }
    return cols;
}

}  // namespace

// Among the z tilings whose buffers fit `cap`: the one that stages the fewest
// volume columns per plane (halo columns are staged once per tile), a tiling
// with several j-blur strips per thread counted half as much again (each
// strip repeats the unrolled blur code with few warps to hide its latency).
// At 192^3 (PSF radius 19) three 64-column tiles with 512 threads beat two
// 96-column tiles with two strips per thread: 1.25 vs 1.51 ms (384 threads)
// and 1.77 ms (288) per launch of 16 angles and two volumes; at 160^3 two
// 80-column tiles beat three of 64, 172 vs 233 us for 8 angles.
// The halo of tiles is a multiple of 4, which keeps a staged window 16-byte
// aligned, or even where no tile fits with that (planes of n = 689 to 720 with
// radius 17 or 18).
PlaneTiling plane_tiling(int n, int nz, int rmax, size_t cap, size_t limit)
{
    PlaneTiling best{};
    double best_cost = 0;
    for (int halo = 4; halo >= 2 && best.smem == 0; halo -= 2)
        for (int nt = 1; nt <= (nz + kStrip - 1) / kStrip; ++nt) {
            const int kt = nt == 1 ? nz : round_up((nz + nt - 1) / nt, kStrip);
            if (nt > 1 && (nt - 1) * kt >= nz) continue;  // same as a smaller count
            const PlaneTiling t = make_tiling(n, nz, rmax, kt, halo, cap, limit);
            if (t.smem == 0) continue;
            const double cost = (double)staged_columns(t, nz) * (t.ipt > 1 ? 1.5 : 1.0);
            if (best.smem == 0 || cost < best_cost) {
                best = t;
                best_cost = cost;
            }
        }
    return best;  // smem == 0: does not fit
}

// The forward's tiling in CTAs of a thread per blur strip (64 at least), several
// to an SM.  A CTA of 256 keeps most of its threads idle in the blur of a short
// plane, which suits a launch of one or two planes a CTA (their staging takes all
// threads); a launch of more is bound by the blurs' throughput.  Taken where four or
// more fit an SM.  Whole projections, us with their reduction, CTAs of that size
// always -> 256 threads -> by launch: 48 x 24, 96 angles 53 -> 67 -> 51, four
// volumes 167 -> 220 -> 161; 64^2 x 24, 48 angles, four volumes 156 -> 185 -> 154; 76
// x 36 the same 230 -> 250 -> 223; with three to an SM (76 x 48) 255 -> 252 -> 260.
// smem 0 where CTAs would not get smaller.
PlaneTiling many_tiling(const PlaneTiling& t)
{
    PlaneTiling m = t;
    m.threads = std::max(64, round_up((t.ktpad / 2) * (t.npad / kStrip), 32));
    if (t.ipt > 1 || m.threads >= t.threads) m.smem = 0;
    return m;
}

// Depth chunks, at most `most`, of a launch whose every chunk is `items` CTAs,
// on a device that holds `slots` CTAs at a time: as many as fill one wave, or,
// where that leaves much of it empty, the fewest whose waves take a sixth less
// depth.  Two 64-column tiles and 48 angles are 96 CTAs on 152 SMs: in one chunk
// two volumes are two waves of the whole depth, in three chunks four waves of a
// third (forward, us): 132 x 128 1609 -> 1084, 160 x 104 2164 -> 1467, 128 x 160
// 1489 -> 1008, 102 x 188 1101 -> 758.  A launch that fills a wave stays as it is.
int depth_chunks(long items, long slots, long most)
{
    if (items >= slots) return 1;
    const long first = std::max<long>(1, std::min(most, slots / items));
    const auto waves = [&](long c) { return (items * c + slots - 1) / slots; };
    long best = first;
    for (long c = first + 1; c <= std::min(most, 4 * first); ++c)
        if (6 * waves(c) * best < 5 * waves(best) * c) best = c;
    return (int)best;
}

// Back blur.  Candidates: for each stride of kBackStrides as many tiles as it
// needs, of equal widths, with the narrowest stride that holds one.  Among those
// that fit: the fewest rounds of strips per plane, a round of 256 threads
// counted half; then the widest tile.  The CTA has 256 threads where a pass over
// a plane has that many strips or fewer and two such CTAs fit an SM, else 512,
// and the attenuation comes through shared memory where a tile is the whole
// plane and the buffer fits.  Measured (one subset, us): 64^3 x 8 angles 256
// threads 14.3, two 32-column tiles of 256 16.3; 96^3 x 12 one tile of 512
// threads 39.8, two of 256 47.2; 128^3 x 15 one tile of 512 87, two of 256 85;
// 160^3 x 8 two tiles of 96 columns 117, three of 64 131, and x 12 two of 96 158, of
// 80 154; 192^3 x 16 x 2 volumes three tiles of 64 columns 338, two of 96 406.  A
// wider stride than the tile needs takes the second CTA or the attenuation
// buffer: 132 x 44 x 15 stride 33 two CTAs 47.4, 65 one of 256 threads 54.5, one of
// 512 51.8; 80 x 96 x 12 stride 49 two CTAs 24.9, 65 one of 256 28.6, one of 512
// 26.7; 190 x 56 x 12 stride 33 with the buffer 103, 65 without 173.  Planes of 129
// to 192 columns whole, with the buffer, where they had been two tiles of up to
// 128 (96 angles, us; in brackets with tiles of any width as before the strides
// were fixed): 57 x 144 308 -> 180 [186], 76 x 160 470 -> 285 [303], 102 x 136 588
// -> 424 [426]; two equal tiles of 80 columns in place of 96 or 128: 145 x 136 1219
// -> 972.
BackTiling back_tiling(int n, int nz, int rmax, bool atten, size_t limit)
{
    BackTiling best{};
    double best_cost = 0.0;
    int last_width = 0;
    const int npad = round_up(n, kStrip), rp = npad / 2, rh = rmax + (rmax & 1);
    for (int widest : kBackStrides) {
        BackTiling t{};
        // as many tiles as this stride needs, of equal widths, with the
        // narrowest stride that holds one
        t.ntiles = (nz + 2 * (widest - 1) - 1) / (2 * (widest - 1));
        t.ktile = t.ntiles == 1 ? nz : round_up((nz + t.ntiles - 1) / t.ntiles, kStrip);
        t.ktpad = round_up(t.ktile, kStrip);
        if (t.ktpad == last_width) continue;
        last_width = t.ktpad;
        for (int i = (int)(sizeof kBackStrides / sizeof kBackStrides[0]) - 1; i >= 0; --i)
            if (2 * (kBackStrides[i] - 1) >= t.ktpad) t.sq = kBackStrides[i];
        t.rh = rh;
        t.npad = npad;
        t.pad_rows = (rmax + 1) / 2;
        t.high = rmax > kLowR;
        t.sp = ((t.ktpad + 2 * rh) / 2) | 1;
        size_t off = 16 * (size_t)rp * t.sp;
        t.off_q = (int)off;
        off += 16 * (size_t)(rp + 2 * t.pad_rows) * t.sq;
        t.off_taps = (int)off;
        off += 2 * kTapRow * sizeof(float);
        const size_t bare = off, a_at = (off + 15) & ~(size_t)15;  // bulk copies land on 16-byte boundaries
        const size_t with_a = a_at + (size_t)n * t.ktile * sizeof(float) + 8;
        t.off_a = (int)a_at;
        t.off_bar = (int)(with_a - 8);
        const int zitems = rp * (t.ktpad / kStrip), jitems = (t.ktpad / 2) * (npad / kStrip);
        t.smem_a = atten && t.ntiles == 1 && with_a <= limit;  // a tile's rows would be copied one by one
        t.smem = t.smem_a ? with_a : bare;
        if (t.smem > limit) continue;
        const bool two = 2 * (t.smem + 1024) <= kSmSmem;
        const int thr = two && std::max(zitems, jitems) <= kPlaneThreads / 2 ? kPlaneThreads / 2 : kPlaneThreads;
        t.threads = thr;
        t.zstep = {thr % rp, thr / rp};
        t.jstep = {thr % (t.ktpad / 2), thr / (t.ktpad / 2)};
        const int rounds = (zitems + thr - 1) / thr + (jitems + thr - 1) / thr;
        const double cost = (double)rounds * thr * t.ntiles;
        if (best.smem == 0 || cost <= best_cost) {
            best = t;
            best_cost = cost;
        }
    }
    return best;  // smem == 0: does not fit
}

int forward_max_blocks_per_sm(const PlaneTiling& t)
{
    switch (t.ipt) {
        case 1: return t.high ? forward_occupancy_ipt<1, true>(t.threads, t.smem) : forward_occupancy_ipt<1, false>(t.threads, t.smem);
        case 2: return forward_occupancy_ipt<2, true>(t.threads, t.smem);
        case 3: return forward_occupancy_ipt<3, true>(t.threads, t.smem);
        default: return forward_occupancy_ipt<4, true>(t.threads, t.smem);
    }
}

cudaError_t launch_forward(const ForwardArgs& a, cudaStream_t st)
{
    switch (a.t.ipt) {
        case 1: return a.t.high ? forward_launch_ipt<1, true>(a, st) : forward_launch_ipt<1, false>(a, st);
        case 2: return forward_launch_ipt<2, true>(a, st);
        case 3: return forward_launch_ipt<3, true>(a, st);
        default: return forward_launch_ipt<4, true>(a, st);
    }
}

int blur_back_max_blocks_per_sm(const BackTiling& t)
{
    if (t.smem_a) return t.high ? blur_back_blocks_v<true, true>(t) : blur_back_blocks_v<true, false>(t);
    return t.high ? blur_back_blocks_v<false, true>(t) : blur_back_blocks_v<false, false>(t);
}

cudaError_t launch_blur_back(const BlurBackArgs& a, cudaStream_t st)
{
    if (a.t.smem_a) return a.t.high ? launch_blur_back_v<true, true>(a, st) : launch_blur_back_v<true, false>(a, st);
    return a.t.high ? launch_blur_back_v<false, true>(a, st) : launch_blur_back_v<false, false>(a, st);
}

}  // namespace spect
