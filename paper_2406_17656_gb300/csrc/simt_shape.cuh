// simt_shape.cuh -- a lane's shared memory in the thread-per-column kernels
// (lsq_simt.cu), as plain constants: the regions, what overlaps what, and the
// bounds of every access, checked when a shape is used.
#pragma once

namespace sam {

constexpr int simt_tri(int q) { return q * (q + 1) / 2; }

constexpr int kSimtWarps = 16;  // one-warp blocks per SM at most (128 registers each)

// One column problem per lane: up to MAXI rows and MAXJ unknowns.  Word i of a
// lane's shared memory is at 32 i + lane, so that any index of any lane hits its
// own bank; all offsets and sizes below are in words of a lane.
template <int MAXI_, int MAXJ_, bool ADJ = false>
struct SimtShape {
    static constexpr int MAXI = MAXI_, MAXJ = MAXJ_;
    static constexpr int ROWS = MAXI + 1;                // and the row of the padding entries
    static constexpr int GW = simt_tri(MAXJ + 1);        // rows 0..MAXJ of [G b], then of L
    // the adjoint's r (FP64, 2 words a row) takes their place at the end
    static constexpr int LW = ((ADJ && 2 * ROWS > GW ? 2 * ROWS : GW) + 3) & ~3;
    static constexpr int RW = LW;                        // r in FP64 (2 words a row)
    static constexpr int NW = 2;                         // columns of [B c] held dense at a time in the Gram pass
    static constexpr int WW = RW;                        // they take r's place (NW words a row)
    static constexpr int TAB = RW + 2 * ROWS;            // columns of J
    static constexpr int XD = (TAB + MAXJ + 1) & ~1;     // the adjoint's FP64 vectors over J (2 x MAXJ)
    static constexpr int WORDS = ADJ ? XD + 4 * MAXJ : TAB + MAXJ;
    // the Gram pass writes G and w; w and r end before the table of columns
    static_assert(GW <= LW && WW >= LW && WW + NW * ROWS <= TAB && RW + 2 * ROWS <= TAB, "regions");
    static_assert(!ADJ || (2 * ROWS <= LW && XD >= TAB + MAXJ), "the adjoint's regions");
    // FP64 words are 8-byte aligned; rows go in pairs, the last one that of b at most
    static_assert(MAXJ % 2 == 1 && RW % 2 == 0 && WW % NW == 0 && XD % 2 == 0, "alignment");
    static constexpr int BYTES = 128 * WORDS;
    static constexpr int FIT = 232448 / (BYTES + 1024);
    static constexpr int WARPS = FIT < kSimtWarps ? FIT : kSimtWarps;  // one-warp blocks per SM
};

// the shapes of size classes 0 and 1
using Simt0 = SimtShape<14, 5>;
using Simt1 = SimtShape<26, 9>;
using Simt0Adj = SimtShape<14, 5, true>;
using Simt1Adj = SimtShape<26, 9, true>;

}  // namespace sam
