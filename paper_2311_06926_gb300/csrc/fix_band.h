// Layout of the fixed-point banded passes (k_fix_band.cu): sizes that the kernels, the set-up and
// the rules of the dispatch share.
#pragma once
#include "fix.h"

namespace shp {

constexpr int kR = 8;              // outputs per thread along the band (rows of a segment)
constexpr int kFixBandHalf = 6;    // largest half width of the limb tables
constexpr int kFixBandLimit = 227 * 1024;   // shared memory a block can have
constexpr int kFixBandThreads = 256;        // most threads of a block

// Half width H >= 1: centred square bands, row r of a segment reads entries r .. r + 2 H of the
// window (2 H + 2 stored, the last one zero). H = 0: rectangular bands (the quadrature tables: several
// points per element), whose segments read at most 8 inputs; every row has all 8.
SHP_HD constexpr int band_row(int H) { return H ? H + 1 : 4; }   // int4 per row
// int4 per segment in shared memory: one more than the rows take, so that lanes on neighbouring
// segments read different banks
SHP_HD constexpr int band_seg(int H) { return kR * band_row(H) + 1; }
SHP_HD constexpr int band_segs(int rows) { return (rows + kR - 1) / kR; }

// Staged x1 lines (shared memory): entry j, -H <= j < 8 segs + H, of a line at
// ((j + H) % 8) S + (j + H) / 8 with S odd, zero outside the line; neighbouring threads (segments)
// then read and write neighbouring words, and no window needs a bound.
SHP_HD constexpr int band_stage_s(int segs, int H) { return (segs + (2 * H + 7) / 8) | 1; }

// shared memory of a block of x1 lines: the operators' limbs and scales, and nline staged lines
constexpr int64_t band_along_smem(int nops, int nline, int segs, int H) {
  return (int64_t)nops * segs * band_seg(H) * 16 + ((nops * segs + 1) & ~1) * 4 +
         (int64_t)nline * kR * band_stage_s(segs, H) * 8;
}

// Whether the passes of operators of b rows fit a block. The limb tables of a whole operator are
// staged for a pass along x1, so a launch grows with the mesh; the largest has two terms and two
// results (three operators, four lines per group of segments). Longer operators keep the FMA
// passes, which stage nothing.
constexpr bool fix_band_fits(int b, int H) {
  const int segs = band_segs(b);
  return H >= 1 && H <= kFixBandHalf && segs <= kFixBandThreads &&
         band_along_smem(3, 4 * (kFixBandThreads / segs), segs, H) <= kFixBandLimit;
}

}  // namespace shp
