// The fixed-point banded passes (k_fix_band.cu): sizes that the kernels, the set-up and the rules of
// the dispatch share, and the arithmetic of a thread, which the host compiles too (for its tests).
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

// shared memory of a block of x1 lines: the operators' limbs, and nline staged lines
constexpr int64_t band_along_smem(int nops, int nline, int segs, int H) {
  return (int64_t)nops * segs * band_seg(H) * 16 + (int64_t)nline * kR * band_stage_s(segs, H) * 8;
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

// ---- arithmetic -------------------------------------------------------------------------------
constexpr int kBandLimb = 29, kBandXBits = 57;   // bits of a limb, of a scaled window entry

SHP_HD void band_mad(long long& c, int a, int b) {
  c += (long long)a * b;
}

// The window's exponent (the biased one of its largest entry; -1 if all are zero; slow set when it
// cannot be scaled) and its entries as limbs: x / 2^(exponent - 1022) 2^57 rounded to
// hi 2^29 + lo, |lo| <= 2^28.
template <int N>
SHP_HD int band_limbs(const double (&x)[N], int2 (&v)[N], bool& slow) {
  unsigned key = 0, low = 0;   // key: the largest exponent and leading bits, one place to the left
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const unsigned m = hi_word(x[k]) << 1;
    key = m > key ? m : key;
    low |= lo_word(x[k]);
  }
  const int e = (int)(key >> 21);
  const bool zero = (key | low) == 0;
  slow = slow || (!zero && (e < (int)kFixMinExp || e > (int)kFixMaxExp));
  const int top = zero ? 4000 : 62 - kBandXBits + e;   // (4000: everything shifts out)
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const unsigned hi = hi_word(x[k]), lo = lo_word(x[k]);
    // the significand with its leading one at bit 62 (an entry without one shifts out)
    const unsigned long long n =
        ((unsigned long long)funnel_left(lo, (hi & 0xfffffu) | 0x100000u, 10) << 32) |
        (lo << 10);
    // one bit more than kept, then rounded (truncated entries would all err towards zero, and that
    // smooth error is what the preconditioner amplifies), the low limb of either sign
    const int sh0 = top - (int)((hi >> 20) & 0x7ffu), sh = sh0 < 63 ? sh0 : 63;
    const unsigned long long t = (n >> sh) + (1ull << kBandLimb) + 1;
    const int h = (int)(t >> (kBandLimb + 1));
    const int l = (int)((unsigned)(t >> 1) - (1u << (kBandLimb - 1)) - ((unsigned)h << kBandLimb));
    const int sg = (int)hi >> 31;
    v[k].x = (h ^ sg) - sg;
    v[k].y = (l ^ sg) - sg;
  }
  return zero ? -1 : e;
}

// Row r of the segment times the window, in units of 2^58 of the product of the two scales, plus hh.
template <int H, int N>
SHP_HD long long band_row_dot(const int4* c, const int2 (&v)[N], int r, long long hh = 0) {
  long long md = 1ll << (kBandLimb - 1);
  const int k0 = H ? r : 0;
#pragma unroll
  for (int q = 0; q < band_row(H); ++q) {
    const int4 w = c[r * band_row(H) + q];
    const int2 a = v[k0 + 2 * q];
    band_mad(hh, a.x, w.x);
    band_mad(md, a.x, w.y);
    band_mad(md, a.y, w.x);
    if (H == 0 || q < H) {   // (entry 2 H + 1 is padding)
      const int2 b = v[k0 + 2 * q + 1];
      band_mad(hh, b.x, w.z);
      band_mad(md, b.x, w.w);
      band_mad(md, b.y, w.z);
    }
  }
  return hh + (md >> kBandLimb);
}

// Scale of a window of zeros (below every other) and from scales to the exponent of a result.
constexpr int kNoScale = -(1 << 20);
constexpr int kBandShift = 2 * kBandLimb - 1022 - kBandXBits;

// The outputs 8 seg .. 8 seg + 7 of one line. load(t, x): the window of term t; c: the operators'
// limbs of the segment, cstep int4 apart; ex(o, r): scale of row r of operator o; put(y, r, value):
// output r of Y (y = 0) or Y2 (1). Returns false, without outputs, if a window cannot be scaled.
// ready(): called once the first window is scaled, before the limbs and scales are read.
template <int H, int NT, bool DUAL, typename Ex, typename Load, typename Ready, typename Put>
SHP_HD bool band_outputs(const int4* c, int cstep, Ex&& ex, Load&& load, Ready&& ready,
                         Put&& put) {
  constexpr int N = kR + 2 * H;
  bool slow = false;
  int2 v[N];
  long long s[kR];   // NT = 2: the first term's sums
  int e0 = 0, e = 0;
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    double x[N];
    load(t, x);
    e = band_limbs<N>(x, v, slow);
    if (t == 0) ready();
    if (t + 1 < NT) {
      e0 = e;
#pragma unroll
      for (int r = 0; r < kR; ++r) s[r] = band_row_dot<H, N>(c, v, r);
      c += cstep;
      continue;
    }
    if (slow) return false;
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      int top = e < 0 ? kNoScale : e + ex(t, r);
      long long y;
      if (NT > 1) {
        // both sums at the larger of the two scales, half a unit added to one that is shifted
        const int en = top, es = e0 < 0 ? kNoScale : e0 + ex(0, r);
        top = es > en ? es : en;
        const int da = top - es < 62 ? top - es : 62, db = top - en < 62 ? top - en : 62;
        y = band_row_dot<H, N>(c, v, r, (1ll << db) >> 1);
        y = ((s[r] + ((1ll << da) >> 1)) >> da) + (y >> db);
      } else {
        y = band_row_dot<H, N>(c, v, r);
      }
      put(0, r, fix_to_double(y, top + kBandShift));
      if (DUAL) {
        const int e2 = e < 0 ? kNoScale : e + ex(NT, r);
        put(1, r, fix_to_double(band_row_dot<H, N>(c + cstep, v, r), e2 + kBandShift));
      }
    }
  }
  return true;
}

}  // namespace shp
