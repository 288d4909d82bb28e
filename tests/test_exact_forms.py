"""The integer forms of the FP64 equilibrium (csrc/lbm_exact.h) against the
compiler's FP64, bit for bit: compiled as plain C++ here, over velocities of
every size below the bound, signs, zeros, subnormals and near-ties."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0807_0602_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#include "lbm_exact.h"
using namespace sc::exact;
static u64 B(double x) { u64 b; std::memcpy(&b, &x, 8); return b; }
int main() {
    std::mt19937_64 r(7);
    std::uniform_real_distribution<double> U(-1, 1);
    long bad = 0, used = 0;
    for (long i = 0; i < 3000000; ++i) {
        double ux, uy;
        switch (i % 7) {
            case 0: ux = U(r) * .2; uy = U(r) * .2; break;
            case 1: ux = std::ldexp(U(r), -(int)(r() % 60)); uy = std::ldexp(U(r), -(int)(r() % 60)); break;
            case 2: ux = std::ldexp(1 + ((double)(r() % 5) - 2) * 0x1p-52, -(int)(r() % 60) - 3);
                    uy = std::ldexp(U(r), -(int)(r() % 1080)); break;
            case 3: ux = (r() & 1) ? 0.0 : -0.0; uy = U(r) * .15; break;
            case 4: ux = (double)(r() % 4096) * 0x1p-15; uy = -(double)(r() % 4096) * 0x1p-15; break;
            case 5: ux = U(r) * 0x1p-26; uy = U(r) * 0x1p-27; break;
            default: { const double a = 0.19764; ux = a * std::cos(U(r) * 4); uy = std::sqrt(a * a - ux * ux) * (r() & 1 ? 1 : -1); }
        }
        volatile double xx = ux * ux, yy = uy * uy;
        volatile double usq = xx + yy, d = ux + uy, e = uy - ux;
        if ((unsigned)(B(usq) >> 32) >= (unsigned)kMaxUsqHigh) continue;
        ++used;
        volatile double b = 1.5 * usq, dd = d * d, ee = e * e;
        const Fix fb = b_of(B(usq));
        volatile double e0 = 1.0 - b;
        bad += rest(fb) != B(e0);
        const double cs[4] = {ux, uy, d, e}, cc[4] = {xx, yy, dd, ee};
        for (int q = 0; q < 4; ++q) {
            volatile double t = 3 * cs[q], s = 4.5 * cc[q];
            volatile double p = 1 + t, m = 1 - t;
            p = p + s; m = m + s;
            p = p - b; m = m - b;
            u64 A, C;
            pair(B(cs[q]), B(cc[q]), fb, A, C);
            bad += A != B(p) || C != B(m);
        }
    }
    std::printf("%ld %ld\n", used, bad);
}
"""


def test_integer_forms_equal_fp64(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    src = tmp_path / "exact.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "exact")
    subprocess.run([gxx, "-O2", "-ffp-contract=off", "-I" + CSRC, str(src), "-o", exe], check=True)
    used, bad = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert used > 2_000_000 and bad == 0
