"""Host-side checks of the FP32 plane kernels' tilings (no GPU): the shapes
that plans are created for, from the tiling functions of libspect itself.

A small program linked to the library prints both tilings of the shapes that
it reads; the bounds are the buffers of csrc/plane_host.cu, restated here.
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2309_01977_gb300")
LIMIT = 227 * 1024    # dynamic shared memory of a CTA
CAP = LIMIT - 2048    # less static shared memory (forward)

PROGRAM = r"""
#include <cstdio>
#include "internal.h"
int main()
{
    int n, nz, r, atten;
    while (std::scanf("%d %d %d %d", &n, &nz, &r, &atten) == 4) {
        const spect::PlaneTiling f = spect::plane_tiling(n, nz, r, CAP, LIMIT);
        const spect::BackTiling b = spect::back_tiling(n, nz, r, atten != 0, LIMIT);
        std::printf("%d %d %d %zu %d %d %d %d %d %zu\n", f.ktile, f.ntiles, f.rh, f.smem, b.ktpad, b.ntiles, b.sq,
                    b.threads, (int)b.smem_a, b.smem);
    }
}
"""
FIELDS = ("f_ktile", "f_ntiles", "f_rh", "f_smem", "ktpad", "ntiles", "sq", "threads", "smem_a", "smem")


@pytest.fixture(scope="module")
def tilings(spect_lib, tmp_path_factory):
    """tilings(shapes): one dict of FIELDS per (n, nz, largest radius, attenuation)."""
    from paper_2309_01977_gb300 import build
    spect_lib.load()
    d = tmp_path_factory.mktemp("tilings")
    src, exe = str(d / "tilings.cu"), str(d / "tilings")
    with open(src, "w") as fh:
        fh.write(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-DCAP=%d" % CAP, "-DLIMIT=%d" % LIMIT, "-I",
                    build.INCLUDE, "-I", build.CSRC, "-o", exe, src, "-L", PKG, "-l:libspect.so", "-Xlinker",
                    "-rpath=" + PKG], check=True)

    def ask(shapes):
        text = "".join("%d %d %d %d\n" % s for s in shapes)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
        return [dict(zip(FIELDS, map(int, line.split()))) for line in out if line]
    return ask


def _up(v, m):
    return -(-v // m) * m


def _smallest_forward(n, r):
    """Bytes of the narrowest forward tile (16 columns, the halo rounded up to even)."""
    rh, rp = _up(r, 2), _up(n, 16) // 2
    return 16 * (rp * ((16 + 2 * rh) // 2 | 1) + 8 * ((2 * rp + 2 * rh) // 2 | 1)) + 32 * n + 2 * 21 * 4


def test_planes_that_fit_are_accepted(tilings):
    shapes = [(n, nz, r, 1) for n in range(560, 1025, 8) for nz in (20, 64, 120) for r in range(13, 21)]
    shapes += [(n, 64, r, 1) for n in range(680, 730) for r in (17, 18)]
    took = refused = 0
    for (n, nz, r, _), t in zip(shapes, tilings(shapes)):
        strips = 8 * (_up(n, 16) // 16)  # of a 16-column tile, at most four to a thread of 512
        fits = _smallest_forward(n, r) <= CAP and strips <= 2048
        assert (t["f_smem"] > 0) == fits, (n, nz, r)
        if fits:
            assert 0 < t["smem"] <= LIMIT and t["f_smem"] <= LIMIT, (n, nz, r)
        took, refused = took + fits, refused + (not fits)
    assert took > 100 and refused > 100


def test_back_tilings_carry_no_padding(tilings):
    """The back blur's stride is the narrowest that holds its tile, its tiles are
    equal, a CTA of 256 threads is one of two that fit an SM, a plane of up to 192
    columns is whole and its attenuation staged where that fits."""
    strides = (9, 17, 33, 49, 65, 81, 97)  # kBackStrides
    shapes = [(n, nz, r, 1) for n in range(32, 193, 3) for nz in range(24, 193, 4) for r in (3, 9, 15, 19)]
    halved = staged = 0
    for (n, nz, r, _), t in zip(shapes, tilings(shapes)):
        assert t["smem"] > 0, (n, nz, r)
        assert t["sq"] == min(s for s in strides if 2 * (s - 1) >= t["ktpad"]), (n, nz, r, t)
        assert t["ktpad"] == _up(-(-nz // t["ntiles"]), 16), (n, nz, r, t)
        assert t["threads"] in (256, 512)
        if t["threads"] == 256:
            assert 2 * (t["smem"] + 1024) <= 228 * 1024, (n, nz, r, t)
            halved += 1
        if n <= 80 and nz <= 192 and r <= 9:
            assert t["ntiles"] == 1, (n, nz, r, t)
        rp, rh = _up(n, 16) // 2, _up(r, 2)
        bare = 16 * (rp * ((t["ktpad"] + 2 * rh) // 2 | 1) + (rp + 2 * ((r + 1) // 2)) * t["sq"]) + 2 * 21 * 4
        fits = t["ntiles"] == 1 and _up(bare, 16) + 4 * n * nz + 8 <= LIMIT
        assert t["smem_a"] == fits, (n, nz, r, t)
        staged += fits
    assert halved > 100 and staged > 100
