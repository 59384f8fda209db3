"""Neighbour indices of a row off the y and z faces (csrc/row_index.cuh),
compiled for the host and enumerated over small boxes: both lattices, walls and
periodic x faces, ragged sides, every lane of every 32-node row (those past its
end read as its last node does).  Each index lies inside the lattice and, where
there is a neighbour, is the neighbour."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2206_11634_gb300", "csrc")

HARNESS = r"""
#include <algorithm>
#include <cstdio>
#include "row_index.cuh"
using namespace lbmmb;

int main() {
    long long lanes = 0, walls = 0, outside = 0, wrong = 0;
    for (int nx : {2, 3, 31, 32, 33, 34, 63, 64, 65})
        for (int ny : {3, 4, 6})
            for (int nz : {3, 5})
                for (int per = 0; per < 2; per++)
                    for (int bx0 = 0; bx0 < nx; bx0 += 32)
                        for (int x = bx0; x < bx0 + 32; x++)
                            for (int y = 1; y < ny - 1; y++)
                                for (int z = 1; z < nz - 1; z++)
                                    for (int e = 0; e < 27; e++) {  // D3Q15's and D3Q19's among them
                                        const int ex = e % 3 - 1, ey = e / 3 % 3 - 1, ez = e / 9 - 1;
                                        const int xl = std::min(x, nx - 1), n = xl + nx * (y + ny * z);
                                        const RowLane r = row_lane(xl, nx, per != 0);
                                        const int at = row_neighbour(n, nx, nx * ny, r, ex, ey, ez);
                                        lanes++;
                                        if (at < 0 || at >= nx * ny * nz) outside++;
                                        int sx = xl - ex;
                                        const bool wall = !per && (sx < 0 || sx >= nx);
                                        if (wall != row_wall(r, ex)) wrong++;
                                        if (wall) {
                                            walls++;
                                            if (at != n) wrong++;
                                            continue;
                                        }
                                        sx = (sx + nx) % nx;
                                        if (at != sx + nx * ((y - ey) + ny * (z - ez))) wrong++;
                                    }
    std::printf("%lld %lld %lld %lld\n", lanes, walls, outside, wrong);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_every_neighbour_index_is_inside(tmp_path):
    src = tmp_path / "row.cpp"
    src.write_text(HARNESS)
    exe = tmp_path / "row"
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wno-unknown-pragmas", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    lanes, walls, outside, wrong = map(int, subprocess.run([str(exe)], check=True, capture_output=True,
                                                           text=True).stdout.split())
    assert lanes > 100000 and walls > 1000
    assert outside == 0 and wrong == 0
