"""The shared memory of the thread-per-column kernels (csrc/simt_shape.cuh, plain
C++): the word of every access that csrc/lsq_simt.cu makes, for every number of
unknowns and rows of both size classes, stays in its region and in the lane's
share of the block.  Compiled and run on the CPU."""
import subprocess

from paper_2406_17656_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "simt_shape.cuh"
using namespace sam;
static int bad = 0;
// words [lo, hi) of one pass: inside [from, to) and the lane's memory
static void in(const char *what, int lo, int hi, int from, int to, int words) {
    if (lo < from || hi > to || lo < 0 || hi > words) {
        std::printf("%s: [%d, %d) outside [%d, %d) of %d\n", what, lo, hi, from, to, words);
        ++bad;
    }
}
template <class SH, bool ADJ>
static void check() {
    const int W = SH::WORDS;
    for (int n = 1; n <= SH::MAXJ; ++n)
        for (int i = 0; i <= SH::MAXI; ++i) {  // MAXI: the padding row
            in("w", SH::WW + SH::NW * i, SH::WW + SH::NW * (i + 1), SH::LW, SH::TAB, W);
            in("r", SH::RW + 2 * i, SH::RW + 2 * (i + 1), SH::LW, SH::TAB, W);
            if (ADJ) in("adjoint r", 2 * i, 2 * (i + 1), 0, SH::LW, W);
        }
    for (int n = 1; n <= SH::MAXJ; ++n) {
        // Gram pass: rows q0, q0 + 1 of [G b] while the dense pair w lives
        for (int q0 = 0; q0 < SH::MAXJ + 1 && q0 < n + 1; q0 += SH::NW)
            for (int c = 0; c < n && c < q0 + SH::NW; ++c)
                for (int t = 0; t < SH::NW; ++t)
                    if (q0 + t >= c && q0 + t <= SH::MAXJ) {
                        const int x = simt_tri(q0) + c + t * q0 + simt_tri(t);
                        in("G", x, x + 1, 0, SH::WW, W);
                        if (x != simt_tri(q0 + t) + c) ++bad;
                    }
        // factor: both rows of a pair up to their diagonals
        for (int q0 = 0; q0 < n + 1; q0 += 2)
            in("L", simt_tri(q0), simt_tri(q0 + 1) + q0 + 2, 0, SH::LW, W);
        in("x", simt_tri(n), simt_tri(n) + n, 0, SH::LW, W);
        in("columns of J", SH::TAB, SH::TAB + n, SH::RW + 2 * SH::ROWS, W, W);
        if (ADJ) in("adjoint vectors", SH::XD, SH::XD + 4 * SH::MAXJ, SH::TAB + SH::MAXJ, W, W);
    }
    if (SH::BYTES != 128 * W || SH::WARPS < 1 || SH::WARPS * (SH::BYTES + 1024) > 233472) ++bad;
}
int main() {
    check<Simt0, false>();
    check<Simt1, false>();
    check<Simt0Adj, true>();
    check<Simt1Adj, true>();
    return bad ? 1 : 0;
}
"""


def test_every_access_is_in_its_region(tmp_path):
    src, exe = tmp_path / "layout.cpp", tmp_path / "layout"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", build.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
