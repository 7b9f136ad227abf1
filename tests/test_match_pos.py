"""The candidate numbers of the retrieval kernels (csrc/match_pos.h) at the largest
buffer they take, on the CPU: every row, lane and element around both ends against
64-bit arithmetic, for each offset from a 16-byte boundary."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <stdio.h>
#include "match_pos.h"
using namespace rs;
static int bad = 0;
#define CHECK(x) do { if (!(x)) { if (bad++ < 5) printf("%s: t %lld al %lld row %lld lane %d k %d\n", #x, t, al, row, lane, k); } } while (0)
static void scan(long long t, long long al) {
    const ScanPos s{(uint32_t)t, (uint32_t)al};
    const long long rows = (t + al + 126) / 128;  // up to the row of position t - 2
    long long row = 0; int lane = 0, k = 0;
    CHECK((long long)s.rows() == rows);
    for (row = 0; row < rows + 4; ++row) {
        if (row == 3 && rows > 8) row = rows - 3;
        for (lane = 0; lane < 32; ++lane) {
            const long long p0 = 128 * row + 4 * lane - al;
            const uint32_t q = s.quad((int)row, lane);
            CHECK(s.whole(q) == (p0 >= 0 && p0 + 3 < t));
            if (s.whole(q)) CHECK((long long)q == p0);
            for (int e = 0; e < 4; ++e) {
                const long long p = p0 + e;
                CHECK(s.in(q + e) == (p >= 0 && p < t));
                if (s.in(q + e)) CHECK((long long)(uint32_t)(q + e) == p && (long long)(int)(q + e) == p);
                for (k = 1; k <= 8 && k <= t; ++k) CHECK(s.end(q + e, k) == (p >= k - 1 && p <= t - 2));
                k = 0;
            }
        }
    }
}
int main() {
    const long long top = kMatMaxTokens, sizes[] = {1, 2, 3, 4, 5, 6, 7, 9, 127, 128, 129, 130, 131, 1000, top - 130, top - 128, top - 4, top - 3, top - 2, top - 1, top};
    for (long long t : sizes)
        for (long long al = 0; al < 4; ++al) scan(t, al);
    for (long long t : sizes) {  // lists of t candidates
        const long long al = 0, rows = (t + 127) / 128;
        const ListPos l{(int)t};
        long long row = 0; int lane = 0, k = 0;
        CHECK((long long)l.rows() == rows);
        for (row = rows > 3 ? rows - 3 : 0; row < rows; ++row)
            for (int o = 0; o < 512; ++o) {  // a warp's rows from this one on
                const long long c = 128 * row + o;
                CHECK(l.in((int)row, o) == (c < t));
                if (l.in((int)row, o)) CHECK(l.number((int)row, o) == c);
            }
    }
    {  // clusters of 16 where the context can run all of the call's at once
        long long t = 0, al = 0, row = 0; int lane = 0, k = 0;
        CHECK(match_cluster(1, 4, 7) == 16 && match_cluster(4, 4, 7) == 16 && match_cluster(5, 4, 7) == 8);
        CHECK(match_cluster(7, 8, 7) == 16 && match_cluster(8, 8, 7) == 8 && match_cluster(4, 8, 3) == 8);
        CHECK(match_cluster(1, 4, 0) == 8 && match_cluster(1, 8, 0) == 8);
    }
    printf("bad %d\n", bad);
    return bad != 0;
}
"""


def test_numbers_at_the_ends_of_a_buffer(tmp_path):
    src = tmp_path / "pos.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "pos")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover", "-I",
                    os.path.join(ROOT, "paper_2511_01282_gb300", "csrc"), str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
