"""Host-side check of the depth chunks of a launch (no GPU), from the library's
own function: never more than allowed, a launch that fills a wave is one chunk,
and no choice leaves a sixth of the depth's time to another number of chunks
that it considers.
"""
import os
import subprocess

import pytest

from test_plane_tiling_cpu import PKG

PROGRAM = r"""
#include <cstdio>
#include "internal.h"
int main()
{
    long items, slots, most;
    while (std::scanf("%ld %ld %ld", &items, &slots, &most) == 3)
        std::printf("%d\n", spect::depth_chunks(items, slots, most));
}
"""


@pytest.fixture(scope="module")
def chunks(spect_lib, tmp_path_factory):
    from paper_2309_01977_gb300 import build
    spect_lib.load()
    d = tmp_path_factory.mktemp("chunks")
    src, exe = str(d / "chunks.cu"), str(d / "chunks")
    with open(src, "w") as fh:
        fh.write(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, "-o", exe, src,
                    "-L", PKG, "-l:libspect.so", "-Xlinker", "-rpath=" + PKG], check=True)

    def ask(triples):
        text = "".join("%d %d %d\n" % t for t in triples)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()
        return [int(v) for v in out]
    return ask


def test_depth_chunks(chunks):
    triples = [(i, s, m) for i in range(1, 400) for s in (152, 304, 1216) for m in (1, 2, 3, 6, 20, 64)]
    for (items, slots, most), c in zip(triples, chunks(triples)):
        assert 1 <= c <= most
        if items >= slots:
            assert c == 1, (items, slots, most)
            continue
        first = max(1, min(most, slots // items))
        cost = lambda k: -(-items * k // slots) / k
        assert first <= c <= 4 * first and cost(c) <= cost(first)
        best = min(cost(k) for k in range(first, min(most, 4 * first) + 1))
        assert best >= cost(c) * 5 / 6 - 1e-12, (items, slots, most, c)
        if (items * first) * 6 >= slots * 5:  # the wave is five sixths full
            assert c == first, (items, slots, most, c)


def test_depth_chunks_of_known_launches(chunks):
    # 128^3 x 15 angles; all 120 of them; two tiles of 48 angles; 64^3 x 8 angles, two CTAs an SM
    assert chunks([(15, 152, 20), (120, 152, 2), (96, 152, 6), (8, 304, 32)]) == [10, 1, 3, 32]
