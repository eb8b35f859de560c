"""The strips that a box is cut into (csrc/strip_plan.h), as plain C++ on the host."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_14742_gb300", "csrc")

CPP = r"""
#include <cstdio>
#include <cstdlib>
#include "strip_plan.h"
int main(int argc, char** argv)
{
    int a[8];
    while (std::scanf("%d %d %d %d %d %d %d %d", a, a + 1, a + 2, a + 3, a + 4, a + 5, a + 6, a + 7) == 8) {
        const lbm::StripPlan p = lbm::strip_plan(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7]);
        const lbm::StripShapeCost s = lbm::strip_shape(a[0], a[1], p.shape);
        const long long strips = lbm::strips_of(a[3], a[4], a[6], s.rows);
        std::printf("%d %d %d %lld %lld\n", p.shape, p.chunk, s.rows, strips,
                    strips * (((long long)a[5] + p.chunk - 1) / p.chunk));
    }
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(CPP)
    exe = str(d / "plan")
    # signed overflow ends the program
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-ftrapv", "-I", CSRC, str(d / "plan.cpp"), "-o", exe])

    def ask(boxes):
        text = "\n".join(" ".join(map(str, b)) for b in boxes)
        r = subprocess.run([exe], input=text, capture_output=True, text=True, timeout=60)
        assert r.returncode == 0
        got = [tuple(map(int, l.split())) for l in r.stdout.splitlines()]
        assert len(got) == len(boxes)
        return got

    return ask


def test_boxes_of_every_shape(plans):
    """Every variant gives a chunk of 1 .. nz planes and a number of strips that fits
    an int, for boxes of up to 2^31 - 2 nodes along any axis."""
    big = (1 << 31) - 2
    dims = [(1, 1, 1), (32, 1, 1), (256, 256, 256), (1, 1, big), (1, 1, (1 << 30) + 10), (1, big, 1), (big, 1, 1),
            (2, 2, (1 << 29) - 1), (1, 1 << 15, (1 << 16) - 1), (46340, 46340, 1)]
    boxes = [(q, st, v, nx, ny, nz, per, 152) for nx, ny, nz in dims for q in (19, 27) for st in range(4)
             for v in range(4 if st == 0 else 16) for per in (0, 1)]
    for box, (shape, chunk, rows, strips, items) in zip(boxes, plans(boxes)):
        nx, ny, nz = box[3:6]
        assert 0 <= shape < (1 if box[1] == 0 else 3) and 1 <= chunk <= nz, box
        assert 30 * strips * rows >= nx * ny or nx == 32, box
        assert 0 < items < (1 << 31) - 8, box


def test_fp32_boxes_take_the_faster_shape(plans):
    """By default two rows or four, whichever was measured the faster by 2% or more."""
    two, four = 2, 4
    boxes = [(19, (256, 256, 256), four), (19, (512, 256, 128), four), (19, (384, 384, 384), four),
             (19, (128, 128, 128), four), (19, (250, 130, 90), two), (19, (96, 96, 96), two), (19, (161, 127, 101), two),
             (27, (256, 256, 256), two), (27, (250, 130, 90), two), (27, (200, 200, 200), four),
             (27, (96, 256, 128), four), (19, (100, 300, 120), four), (19, (160, 160, 160), four), (27, (320, 320, 320), two)]
    got = plans([(q, 1, 0, *d, 1, 152) for q, d, _ in boxes])
    assert [rows for _, _, rows, _, _ in got] == [rows for _, _, rows in boxes]


def test_compact_strips_are_cut_where_they_are_few(tmp_path):
    """Strips of whole tile columns (24 or 32 planes) only where they fill the GPU; a
    part always divides the column. The list waits for strips that fill it more than
    once."""
    (tmp_path / "c.cpp").write_text(r"""
#include <cstdio>
#include <initializer_list>
#include "strip_plan.h"
int main()
{
    for (int q : {19, 27})
        for (int st = 0; st < 4; ++st)
            for (int z : {24, 32})
                for (long long n : {1ll, 100ll, 1000ll, 3000ll, 100000ll, 1ll << 30})
                    for (long long l : {1000ll, 10000000ll}) {
                        const lbm::CompactPlan p = lbm::compact_plan(q, st, 0, z, n, l, 152);
                        std::printf("%d %d %lld %lld %d %d\n", st, z, n, l, p.planes, (int)p.first);
                    }
}
""")
    exe = str(tmp_path / "c")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-ftrapv", "-I", CSRC, str(tmp_path / "c.cpp"), "-o", exe])
    for line in subprocess.check_output([exe], text=True).splitlines():
        st, z, n, listed, part, first = map(int, line.split())
        assert 4 <= part <= z and z % part == 0
        assert part < z if n <= 100 else (n < 100000 or part == z), line
        assert first == (1 if n <= 100 and (st >= 2 or listed == 1000) else 0) or 100 < n < 100000, line
