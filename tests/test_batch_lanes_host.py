"""Streams of a batch's systems (batch_lanes.h): a polymer never shares one, systems that find SMs run
side by side, and queueing never makes the estimated end later than all side by side."""
import os
import subprocess

import paper_1312_2213_gb300._build as build

SRC = r"""
#include <cstdio>
#include <random>
#include "batch_lanes.h"
using namespace muca;
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
static std::vector<int> own_lanes(size_t n) { std::vector<int> o; for (size_t i = 0; i < n; ++i) o.push_back((int)i); return o; }
int main()
{
    const int nsm = 152;
    // three equal systems of 100 blocks, one an SM: two waves side by side, three rounds in one queue
    std::vector<LaneSystem> three(3, LaneSystem{100, 1, 1.0, false});
    CHECK(lanes_end(three, {0, 1, 2}, nsm) == 2.0 && lanes_end(three, {0, 0, 0}, nsm) == 3.0);
    CHECK(lanes_end(three, plan_lanes(three, nsm), nsm) == 2.0);
    // the nine systems of the mix with 2048 walkers: the light ones queue, the end is the heaviest's
    std::vector<LaneSystem> mix = {{32, 1, 4096, false}, {64, 1, 2765, false}, {32, 1, 2304, false}, {32, 1, 1229, false},
                                   {32, 2, 1024, false}, {32, 1, 691, false}, {32, 2, 576, false}, {32, 1, 307, false},
                                   {32, 2, 256, false}};
    const std::vector<int> m = plan_lanes(mix, nsm);
    CHECK(m[0] == 0 && m[1] == 1 && m[2] == 2 && m[3] == 3);
    for (int r = 4; r < 9; ++r) CHECK(m[r] <= 5 && m[r] > 0);
    CHECK(lanes_end(mix, m, nsm) == 4096.0);
    // lattices that overfill the SMs, with polymers between them
    std::vector<LaneSystem> crowd = {{160, 1, 164, false}, {0, 1, 130, true}, {160, 1, 123, false}, {0, 1, 77, true},
                                     {32, 1, 50, false}};
    std::mt19937 g(1);
    for (int trial = 0; trial < 3000; ++trial) {
        std::vector<LaneSystem> s = crowd;
        if (trial) {
            s.clear();
            const int n = 1 + (int)(g() % 12);
            for (int i = 0; i < n; ++i) {
                const bool poly = g() % 4 == 0;
                s.push_back({poly ? 0 : 1 + (int)(g() % (g() % 3 ? 200 : 700)), 1 + (int)(g() % 4), 1.0 + g() % 50, poly});
            }
            std::stable_sort(s.begin(), s.end(), [](const LaneSystem &a, const LaneSystem &b) { return a.cost > b.cost; });
        }
        const std::vector<int> l = plan_lanes(s, nsm);
        CHECK(l.size() == s.size());
        for (size_t r = 0; r < s.size(); ++r) {
            CHECK(l[r] >= 0 && l[r] < (int)s.size());
            for (size_t q = 0; q < s.size(); ++q) CHECK(q == r || l[q] != l[r] || (!s[q].polymer && !s[r].polymer));
        }
        CHECK(lanes_end(s, l, nsm) <= lanes_end(s, own_lanes(s.size()), nsm));
    }
    return 0;
}
"""


def test_lanes(tmp_path):
    src, exe = tmp_path / "lanes.cpp", tmp_path / "lanes"
    src.write_text(SRC)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-Wall", "-I", build.CSRC, str(src),
                           "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
