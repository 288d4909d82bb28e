"""Item numbers of chained launches (csrc/lbm_chain_items.h): every launch of a
long interval keeps them within 32 bits, whatever the number of steps and
tiles, and the numbers map to every tile of every step once."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0807_0602_gb300", "csrc")

HARNESS = r"""
#include <algorithm>
#include <climits>
#include <cstdio>
#include <set>
#include <vector>
#include "lbm_chain_items.h"
using namespace sc;
int main() {
    long bad = 0, launches = 0;
    const long long ctas = 152 * 32;   // each draws one number beyond the last item
    for (long long nt : {1LL, 3LL, 456LL, 1330LL, 10240LL, 10640LL, 68096LL, 1LL << 20, 1LL << 25, 1LL << 29, (1LL << 31) - 1})
        for (long long n : {1LL, 2LL, 50LL, 31537LL, 209716LL, 1900000LL, 1LL << 31}) {
            // the first launches and the last one (all between are alike)
            long long left = n;
            for (int k = 0; k < 4 && left > 0; ++k) {
                const long long m = chain_launch_steps(left, nt, 1);
                ++launches;
                bad += m < 1 || m > left || (m > 1 && m * nt + ctas > INT_MAX);
                bad += m < left && (m + 1) * nt <= kChainItems && m + 1 <= kChainNodeSteps;   // no shorter than need be
                if (m > 1 && m * nt + ctas <= INT_MAX) {
                    // the tiles of the highest and of the drawn-beyond numbers, in runs of `per` tiles
                    for (long long per : {nt, (nt + 2) / 3})
                        for (int rot : {1, 2, 1023})
                            for (long long item : {0LL, nt - 1, m * nt - 1, m * nt / 2, m * nt, m * nt + ctas}) {
                                int step;
                                const int t = chain_item_tile((int)item, (int)nt, (int)m, rot, [&](int i, int& f, int& c) {
                                    f = (int)(i / per * per);
                                    c = (int)std::min(per, nt - f);
                                }, step);
                                bad += item < m * nt ? (t < 0 || t >= nt || step != item / nt) : t != -1;
                            }
                }
                left -= m;
            }
        }
    // the length of a launch: 2^25 nodes times steps, or 8 steps of a larger grid
    for (long long nodes : {1LL, 30000LL, 266240LL, 1310720LL, 5000000LL, 67108864LL, 1LL << 30})
        for (long long n : {1LL, 7LL, 8LL, 25LL, 50LL, 1000LL, 100000000LL}) {
            const long long nt = nodes / 62 + 1, m = chain_launch_steps(n, nt, nodes);
            bad += m < 1 || m > n || (m > 8 && m * nodes > (1LL << 25));
            bad += m < n && m < 8 && nt * 8 <= kChainItems;
            bad += n * nodes <= (1LL << 25) && n * nt <= kChainItems && m != n;
        }
    // every tile of every step once
    for (int nt : {1, 2, 7, 40})
        for (int per : {1, 3, 40})
            for (int rot : {1, 2, 5, 1023})
                for (int step = 0; step < 9; ++step) {
                    std::set<int> seen;
                    for (int i = 0; i < nt; ++i) {
                        int s;
                        seen.insert(chain_item_tile(step * nt + i, nt, 9, rot, [&](int j, int& f, int& c) {
                            f = j / per * per;
                            c = std::min(per, nt - f);
                        }, s));
                        bad += s != step;
                    }
                    bad += (int)seen.size() != nt || *seen.begin() != 0 || *seen.rbegin() != nt - 1;
                }
    std::printf("%ld %ld\n", launches, bad);
}
"""


def test_item_numbers_stay_in_range(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    src = tmp_path / "items.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "items")
    subprocess.run([gxx, "-O2", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover", "-I" + CSRC, str(src),
                    "-o", exe], check=True)
    launches, bad = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert launches > 50 and bad == 0


def test_every_chained_launch_goes_through_the_bound():
    """One place issues chained launches, and it asks for the bound."""
    text = open(os.path.join(CSRC, "lbm_capi.cu")).read()
    assert text.count("L.chain(") == 1
    body = text.split("cudaError_t issue_chain(", 1)[1].split("\n}\n", 1)[0]
    assert "L.chain(" in body and "chain_launch_steps(" in body
