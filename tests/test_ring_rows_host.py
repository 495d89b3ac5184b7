"""Row counters of the sweep's hand-over rings at any number of sweeps: no chunk overflows a 32-bit
counter, and slot, phase and the left-out row of the test hook stay those of a 64-bit count."""
import os
import subprocess

import paper_1312_2213_gb300._build as build

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "ring_rows.h"
using namespace muca;
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main()
{
    const int sizes[] = {8, 12, 16, 24, 32, 48, 64}, blocks[] = {32, 64, 256}, depths[] = {2, 4};
    const int64_t counts[] = {1, 7, 300000000, int64_t(1) << 40, INT64_MAX};
    for (int L : sizes)
        for (int block : blocks)
            for (int record = 0; record < 2; ++record)
                for (int64_t sweeps : counts) {
                    const uint64_t cap = 0xFFFFFFFFull / ((uint64_t)block * (record ? 1 : L * L));
                    const int n = chunk_sweeps(cap, sweeps, L);
                    CHECK(n >= 1 && n <= sweeps && (uint64_t)n <= cap);
                    CHECK((int64_t)n * L + 8 <= INT32_MAX);
                    // nothing smaller than what any of the three bounds asks for
                    CHECK(n == sweeps || (uint64_t)n == cap || (int64_t)(n + 1) * L > kMaxChunkRows);
                }
    CHECK(chunk_sweeps(3, 10, 8) == 3 && chunk_sweeps(0, 10, 8) == 1);
    const int64_t drops[] = {-1, 0, 5, 12, (1 << 30) - 1, 1 << 30, (1 << 30) + 13, INT32_MAX};
    const int64_t chunks[] = {12, 8, 1, 3, 1 << 30, (1 << 30) - 4, 36, 1 << 30, 1 << 30, 1 << 30};
    for (int depth : depths)
        for (int64_t d : drops) {
            int k = 0, drop = (int)d;
            int64_t row = 0;  // rows so far
            for (int64_t n : chunks) {
                CHECK(k % depth == row % depth && (k / depth) % 2 == (row / depth) % 2 && k >= 0 && k < 2 * depth);
                // the hook's row lies in this chunk for both counts or for none, at the same place
                const bool want = d >= row && d < row + n, got = drop >= k && drop < k + n;
                CHECK(want == got);
                if (want) CHECK(drop - k == d - row);
                k += (int)n;
                row += n;
                rebase_rows(k, drop, depth);
            }
        }
    return 0;
}
"""


def test_row_counters(tmp_path):
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(SRC)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-Wall", "-I", build.CSRC, str(src),
                           "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
