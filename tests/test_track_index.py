"""Index arithmetic of the tracking kernel (csrc/track_index.cuh), compiled for the host.

The groups of a warp reduce at different times and in two kinds: 16 sums in rows of
their lanes, 4 sums in a denser layout. A group's lanes synchronise among themselves
only, so both kinds must stay inside the group's own rows."""
import math
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_09971_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "track_index.cuh"
int main()
{
    for (int G : {8, 16, 32})
        for (int wl = 0; wl < 32; ++wl) {
            const int lane = wl & (G - 1);
            std::printf("%d %d %d %d", G, wl, dgf::kRowStride, dgf::short_read(wl, lane));
            for (int i = 0; i < 4; ++i) std::printf(" %d", dgf::short_place(wl, lane, i));
            std::printf("\n");
        }
}
"""


def run_host(tmp_path, program):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(program)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout


def test_short_reduction_stays_in_the_groups_rows(tmp_path):
    rows = [tuple(map(int, line.split())) for line in run_host(tmp_path, PROGRAM).splitlines()]
    assert len(rows) == 96
    for G in (8, 16, 32):
        mine = {wl: (stride, read, place) for g, wl, stride, read, *place in rows if g == G}
        for wl, (stride, read, place) in mine.items():
            g0, lane = wl & ~(G - 1), wl & (G - 1)
            own = range(stride * g0, stride * (g0 + G))
            assert all(p in own for p in place) and read in own and read + 3 in own
            # four places of one value: lanes 4 (lane / 4) .. + 3 of the group, a 16-byte read
            assert read % 4 == 0
            first = g0 + 4 * (lane // 4)
            assert [read + j for j in range(4)] == [mine[first + j][2][lane & 3] for j in range(4)]
        places = [p for _, _, place in mine.values() for p in place]
        assert len(set(places)) == len(places)
        for i in range(4):  # stores of one value and reads of eight lanes: no bank conflicts
            assert len({place[i] % 32 for _, _, place in mine.values()}) == 32
        for q in range(0, 32, 8):
            assert len({mine[wl][1] % 32 // 4 for wl in range(q, q + 8)}) == 8


FAR = r"""
#include <cstdio>
#include <initializer_list>
#include <limits>
#include "track_index.cuh"
int main()
{
    const float inf = std::numeric_limits<float>::infinity(), nan = std::numeric_limits<float>::quiet_NaN();
    for (int R : {1, 4, 5, 7})
        for (int n : {16, 17, 375, 8192})
            for (float f : {0.f, 3.f, -3.f, -20.f, -63.f, -64.f, -65.f, 12.f, n - 1.f, n + 4.f, n + 63.f, n + 64.f, n + 65.f, 1e5f,
                            -1e5f, 2147483520.f, 2147483648.f, -2147483648.f, -2147483904.f, 3e9f, -3e9f, 1e38f, -1e38f, inf,
                            -inf, nan}) {
                const int b = dgf::tap_origin(f, R, n);
                std::printf("%d %d %.9g %d %d\n", R, n, f, b, (int)dgf::taps_inside(b, 2 * R + 3, n, 12));
            }
}
"""


def test_taps_of_points_anywhere(tmp_path):
    """The taps of a point far outside the level, infinite or NaN are read clamped, and no
    index leaves int's range; those of any other point are where exact arithmetic puts
    them, up to taps that clamp to the same border pixel."""
    lines = run_host(tmp_path, FAR).splitlines()
    assert len(lines) == 4 * 4 * 26
    for line in lines:
        R, n, f, b, inside = (float(v) if i == 2 else int(v) for i, v in enumerate(line.split()))
        assert -(1 << 20) < b < 1 << 20
        taps = range(b, b + 2 * R + 3)
        if math.isfinite(f):
            exact = int(f) - R
            clamp = lambda x: min(max(x, 0), n - 1)
            assert [clamp(x) for x in taps] == [clamp(x) for x in range(exact, exact + 2 * R + 3)]
            assert inside == (exact >= -12 and exact + 2 * R + 2 <= n + 11)
        else:
            assert not inside
