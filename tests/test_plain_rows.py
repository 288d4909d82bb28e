"""The plain rows of the bidirectional march (plain_rows in csrc/lbm_device.h):
a row counts as plain only where no node of the tile's columns or of their
neighbours, periodic in both directions, is solid and nothing wraps in y.
Compiled as plain C++ here and compared with the solid nodes themselves for
every tile of many grids, among them those whose last strip is one column
wide with plates at column 0 only."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0807_0602_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <vector>
#include "lbm_device.h"
int main() {
    long rows = 0, plain = 0, wrong = 0;
    for (int W : {64, 128})
        for (int nx = 1; nx <= 400; ++nx)
            for (int ny : {1, 2, 3, 9, 24})
                for (int c = 0; c < 7; ++c) {
                    const int caps[7][2] = {{0, nx / 3}, {0, 1}, {0, nx}, {nx / 3, nx}, {nx / 4, nx / 2},
                                            {nx - 1, nx}, {nx / 2, nx / 2}};
                    const int cx0 = caps[c][0], cx1 = caps[c][1], yb = ny > 2 ? 1 : -1, yt = ny - 2 > yb ? ny - 2 : -1;
                    auto solid = [&](int x, int y) {
                        x = (x % nx + nx) % nx;
                        y = (y % ny + ny) % ny;
                        return x >= cx0 && x < cx1 && (y == yb || y == yt);
                    };
                    for (int R : {1, 5, 24})
                        for (int x0 = 0; x0 < nx; x0 += W - 2)
                            for (int y0 = 0; y0 < ny; y0 += R) {
                                const int ncols = W - 2 < nx - x0 ? W - 2 : nx - x0, y1 = y0 + R < ny ? y0 + R : ny;
                                int first, count;
                                sc::plain_rows(sc::Tile{0, x0, y0, y1}, ncols, nx, ny, cx0, cx1, yb, yt, false, first,
                                               count);
                                rows += y1 - y0;
                                plain += count;
                                for (int r = first; r < first + count; ++r) {
                                    bool ok = nx >= 4 && r >= y0 - 1 && r <= y1 && r >= 1 && r <= ny - 2;
                                    for (int x = x0 - 2; x <= x0 + ncols + 1; ++x)
                                        for (int d = -1; d <= 1; ++d) ok = ok && !solid(x, r + d);
                                    wrong += !ok;
                                }
                                sc::plain_rows(sc::Tile{0, x0, y0, y1}, ncols, nx, ny, cx0, cx1, yb, yt, true, first,
                                               count);
                                wrong += count != 0;
                            }
                }
    std::printf("%ld %ld %ld\n", rows, plain, wrong);
}
"""


def test_plain_rows_have_no_solid_neighbour(tmp_path):
    gxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if gxx is None or not os.path.exists(nvcc):
        pytest.skip("g++ or the CUDA headers not found")
    inc = os.path.realpath(os.path.join(os.path.dirname(os.path.realpath(nvcc)), "..", "include"))
    src = tmp_path / "plain.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "plain")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I" + inc, "-I" + os.path.join(ROOT, "include"), "-I" + CSRC, str(src),
                    "-o", exe], check=True)
    rows, plain, wrong = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert wrong == 0
    assert plain > rows // 4   # and most rows away from the plates are plain
