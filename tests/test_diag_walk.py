"""Index arithmetic of the diagonal product (csrc/diag_walk.h), compiled for the CPU
with overflow checks: every chunk of 32 rows is taken by exactly one warp, whatever
the grid, tiles and number of chunks (whole rounds, none, and several of them), and
a chunk past the end has no row below n, also where 32 times its number leaves an int."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstdint>
#include <cstdio>
#include <vector>
#include "diag_walk.h"
using namespace rbs;
static long fails = 0;
template <int T> static void cover(int begin, int chunks, int nblk, int nw) {
    std::vector<int> taken((size_t)chunks, 0);
    for (int blk = 0; blk < nblk; blk++)
        for (int wid = 0; wid < nw; wid++) {
            const DiagChunks<T> d{begin, begin + chunks, blk, nblk, wid, nw};
            int steps = 0;
            for (auto w = d.first(); w.c < d.end; w = d.next(w)) {
                if (w.c < begin || ++steps > chunks) { fails++; break; }
                taken[(size_t)(w.c - begin)]++;
            }
        }
    for (int t : taken) fails += t != 1;
}
template <int T> static void edge(int64_t n, int begin, int nblk, int nw) {
    const int end = (int)((n + 31) / 32);
    for (int blk : {0, nblk / 2, nblk - 1})
        for (int wid : {0, nw - 1}) {
            const DiagChunks<T> d{begin, end, blk, nblk, wid, nw};
            auto w = d.first();
            for (int past = 0; past < 3; past += w.c >= end, w = d.next(w))
                for (int lane : {0, 31}) {
                    const int64_t want = (int64_t)w.c * 32 + lane;
                    const unsigned got = d.row(w.c, lane);
                    fails += w.c < end ? got != want : got < n;
                }
        }
}
int main() {
    for (int nblk : {1, 3, 152, 456})
        for (int nw : {1, 4, 8})
            for (int chunks : {0, 1, 31, 500, 7295, 7296, 7297, 14600, 22000})
                for (int begin : {0, 64}) { cover<1>(begin, chunks, nblk, nw); cover<4>(begin, chunks, nblk, nw); }
    for (int64_t n : {(int64_t)0x7fffffff, (int64_t)0x7fffffff - 500, (int64_t)0x7fffffff - 31, (int64_t)1 << 30})
        for (int nblk : {1, 456}) {
            const int begin = (int)(n / 32) - 3000;
            edge<1>(n, begin, nblk, 8);
            edge<4>(n, begin, nblk, 4);
        }
    printf("%ld\n", fails);
    return 0;
}
"""


def test_every_chunk_once_and_no_row_past_the_end(tmp_path):
    src, exe = tmp_path / "walk.cpp", tmp_path / "walk"
    src.write_text(SRC)
    csrc = os.path.join(ROOT, "paper_2302_04180_gb300", "csrc")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover", f"-I{csrc}", str(src),
                        "-o", str(exe)], capture_output=True, text=True)
    if r.returncode and "sanitize" in r.stderr:
        pytest.skip("no undefined-behaviour checks in this compiler")
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout + r.stderr
